// FSI cycles of a small image in one cooperative launch: the register-blocked FP32 step
// (step_fast.cuh) with every tile resident for all steps.
//
// A CTA keeps its tile's window, u^{k-1} and mask in shared memory and registers; after a
// step only the pixels other tiles need travel. Every such pixel is published as one
// 64-bit word (value, tag of the step) with a relaxed store, and a tile gathers the halo
// of its window by polling those words until their tags are the step's: value and tag
// arrive together, so no fence, no flag and no second round trip is needed. Two images of
// words, by the parity of the step, are enough: a tile publishes step k + 2 only after it
// has gathered step k + 1 from all its neighbours, each of which published that after
// gathering step k.
//
// The change of a cycle is summed by the last tile to arrive at its end, which stores the
// verdict; nobody waits for it there. A tile looks at the verdict of cycle m at the end of
// cycle m + 1, and if that says stop, the iterate of cycle m is still in its buffer: the
// two buffers take the ends of the cycles in turn.
//
// Bound: latency. What this saves is the launch, the dependency on the previous grid and the
// window load of every step (about 3.3 us of a 512 x 512 step's 5.6). A 256 x 256 step on
// 64 x 8 tiles (R = 3) takes 2.57 us; by clocks in the kernel when it took 2.71: x pass 0.13,
// y pass 0.14, tensor 0.36, divergence and update 0.27, halo exchange 1.4 (a store and a load
// through the L2, 1.0 by itself, plus the wait for the slowest neighbour), the change of the
// cycle 0.08. Before: 4.5 us, one launch per step. A cooperative launch costs some 25 us, hence many cycles in
// one (2.9 us a step with one launch per cycle of 25).
//
// It fits when all tiles are resident at once, which the cooperative launch guarantees.
// Waits are bounded (kPollLimit): a tile that does not see a tag in time raises ctl->timeout
// and leaves, and so do the others; the caller then runs the step kernels.
#pragma once

#include "step_fast.cuh"

namespace foeed {

__device__ __forceinline__ void halo_store(unsigned long long *d, const float v, const uint32_t tag)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(d), "l"(((unsigned long long)tag << 32) | __float_as_uint(v))
                 : "memory");
}
__device__ __forceinline__ void halo_store2(unsigned long long *d, const float a, const float b, const uint32_t tag)
{
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(d), "l"(t | __float_as_uint(a)),
                 "l"(t | __float_as_uint(b))
                 : "memory");
}
__device__ __forceinline__ unsigned long long halo_load(const unsigned long long *s)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(s) : "memory");
    return v;
}
__device__ __forceinline__ void halo_load2(const unsigned long long *s, unsigned long long &a, unsigned long long &b)
{
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(s) : "memory");
}

// The halo of a tile's window in pixel pairs: HL rows above and below, HE columns (HL
// rounded up to a pair) left and right.
template <int R, int TH, int NTHR>
struct CycleHalo {
    static constexpr int HL = R + 2, HE = (HL + 1) & ~1;
    static constexpr int NP = (64 + 2 * HE) / 2;              // pairs of a row above or below
    static constexpr int EDGE = 2 * HL * NP;
    static constexpr int NI = EDGE + TH * HE;                 // pairs in all
    static constexpr int K = (NI + NTHR - 1) / NTHR;          // of one thread
};

__device__ __forceinline__ int reflect(const int i, const int n)
{
    return i < 0 ? -1 - i : (i >= n ? 2 * n - 1 - i : i);
}

// What one thread gathers of a tile's halo: word offsets (o1 negative: one pixel), window
// index of the first pixel, and which of the K entries are used.
template <int K>
struct HaloItems {
    int o0[K], o1[K], dst[K];
    uint32_t used;
};

// The halo of the tile at (x0, y0), whose part inside the image is we x he.
template <int SU_W, typename H, int NTHR>
__device__ __forceinline__ void halo_items(HaloItems<H::K> &q, const int w, const int h, const int pitch, const int x0,
                                           const int y0, const int we, const int he)
{
    q.used = 0;
#pragma unroll
    for (int j = 0; j < H::K; ++j) {
        const int i = threadIdx.x + j * NTHR;
        int r, c;  // window row; column relative to the tile
        if (i < H::EDGE) {
            const int n = i / H::NP;
            c = 2 * (i - n * H::NP) - H::HE;
            r = n < H::HL ? n : n + he;
        } else {
            const int n = (i - H::EDGE) / H::HE, s = i - H::EDGE - n * H::HE;  // HE / 2 pairs on either side
            r = H::HL + n;
            c = s < H::HE / 2 ? 2 * s - H::HE : we + 2 * s - H::HE;
            if (n >= he) c = we + H::HE;
        }
        if (i < H::NI && c < we + H::HE) q.used |= 1u << j;
        const int row = reflect(y0 - H::HL + r, h) * pitch;
        q.o0[j] = row + reflect(x0 + c, w);
        q.o1[j] = c + 1 < we + H::HE ? row + reflect(x0 + c + 1, w) : -1;
        q.dst[j] = r * SU_W + 8 + c;
    }
}

// Gathers them from the words of step `tag` into su; false if a wait ran out.
template <int K>
__device__ __forceinline__ bool gather_halo(const HaloItems<K> &q, const unsigned long long *halo, const uint32_t tag,
                                            float *su, const Ctl *ctl, const int poll0)
{
    uint32_t pend = q.used;
    for (int it = poll0; pend; ++it) {
        unsigned long long a[K], b[K];
#pragma unroll
        for (int j = 0; j < K; ++j)
            if (pend >> j & 1) {
                if (q.o1[j] == q.o0[j] + 1 && !(q.o0[j] & 1)) {
                    halo_load2(halo + q.o0[j], a[j], b[j]);
                } else {
                    a[j] = halo_load(halo + q.o0[j]);
                    b[j] = q.o1[j] >= 0 ? halo_load(halo + q.o1[j]) : a[j];
                }
            }
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((pend >> j & 1) && (uint32_t)(a[j] >> 32) == tag && (uint32_t)(b[j] >> 32) == tag) {
                su[q.dst[j]] = __uint_as_float((uint32_t)a[j]);
                if (q.o1[j] >= 0) su[q.dst[j] + 1] = __uint_as_float((uint32_t)b[j]);
                pend &= ~(1u << j);
            }
        if ((it & 1023) == 1023 && (it >= kPollLimit || *(volatile const int *)&ctl->timeout)) return false;
    }
    return true;
}

// The tile's sums of one cycle's change (cycle number `cycle` of the solve, from 1). The
// last of the ntiles tiles to arrive adds them up in tile order, updates the control block
// as finish_cycle_residual does, and stores the verdict.
__device__ __forceinline__ void cycle_change(double rnum, double rden, Ctl *ctl, double *partials, const int ntiles,
                                             const int bid, const int cycle, double *red)
{
    double *const mine = partials + (cycle & 1) * 2 * ntiles;
    if (grid_sum2_last(rnum, rden, mine, &ctl->arrived[cycle & 1], ntiles, bid, red)) {
        const double rel = rden > 0.0 ? sqrt(rnum) / sqrt(rden) : sqrt(rnum);
        ctl->last_num = rnum;
        ctl->last_den = rden;
        ctl->last_rel = rel;
        ctl->cycles = cycle;
        if (!isfinite(rel)) { ctl->diverged = 1; ctl->done = 1; }
        else if (ctl->tol > 0.0 && rel < ctl->tol) ctl->done = 1;
        __threadfence();
        *(volatile int *)&ctl->verdict[cycle & 1] = ctl->done ? -cycle : cycle;
    }
}

// Whether the solve goes on after cycle number `cycle`; waits for that verdict. A wait that
// runs out raises *dead and stops.
__device__ __forceinline__ bool cycle_goes_on(Ctl *ctl, const int cycle, int *dead, const int poll0)
{
    __shared__ int s_on;
    __syncthreads();
    if (threadIdx.x == 0) {
        int v = 0;
        for (int it = poll0;; ++it) {
            v = *(volatile const int *)&ctl->verdict[cycle & 1];
            if (v == cycle || v == -cycle) break;
            if (it >= kPollLimit || ((it & 1023) == 1023 && *(volatile const int *)&ctl->timeout)) {
                *(volatile int *)&ctl->timeout = 1;
                *dead = 1;
                v = -1;
                break;
            }
        }
        s_on = v > 0;
    }
    __syncthreads();
    return s_on != 0;
}

template <int R, bool EED, typename U, int TH, int LAT, bool VAR>
__global__ void __launch_bounds__(FastTile<R, EED, TH, LAT>::NTHR, FastTile<R, EED, TH, LAT>::MINB)
    fsi_cycle_fast(const __grid_constant__ CycleArgs a)
{
    using G = FastTile<R, EED, TH, LAT>;
    using H = CycleHalo<R, TH, G::NTHR>;
    constexpr int ER = G::ER;
    extern __shared__ __align__(16) float sm[];
    __shared__ double red[64];
    __shared__ int s_dead;
    const StepArgs<float> &p = a.s;
    if (p.ctl->done) return;
    float *su = sm, *sx = su + G::SU_W * G::SU_H, *ss = sx + G::SXT;
    const int tid = threadIdx.x, w = p.w, h = p.h, pitch = (int)p.pitch;
    const int x0 = blockIdx.x * 64, y0 = blockIdx.y * TH;
    const int we = min(64, w - x0), he = min(TH, h - y0);
    const int ntiles = gridDim.x * gridDim.y, bid = blockIdx.y * gridDim.x + blockIdx.x;
    const int cycle0 = p.ctl->cycles;  // cycles of the solve before this launch
    uint32_t tag = (uint32_t)cycle0 * (uint32_t)a.n;
    if (tid == 0) s_dead = 0;
    tile_window<R, EED, TH, LAT>(a.u[0], w, h, pitch, x0, y0, su);
    tile_window_wait();
    const int qe = tid % 16, re = ER * (tid / 16);  // the thread's output groups (tile_divergence)
    float prev[ER][4];
    uint32_t mk[ER];
#pragma unroll
    for (int e = 0; e < ER; ++e) {
        const int r = min(re + e, TH - 1);
        const float4 v = *reinterpret_cast<const float4 *>(su + (r + G::HL) * G::SU_W + 4 * qe + 8);
        prev[e][0] = v.x; prev[e][1] = v.y; prev[e][2] = v.z; prev[e][3] = v.w;
        mk[e] = 0u;  // the internal mask's pitch is a multiple of 32: whole groups lie inside its rows
        if (re + e < TH && y0 + re + e < h && x0 + 4 * qe < w)
            mk[e] = __ldg(reinterpret_cast<const unsigned int *>(p.mask + (long)(y0 + re + e) * pitch + x0 + 4 * qe));
    }
    // the gather's addresses are worked out once, also where they take registers that spill (us a
    // step, per step -> once: 256 x 256 2.71 -> 2.57, 512 x 512 3.76 -> 3.56; 700 x 700, four tiles
    // per SM, 5.68 -> 5.41, sigma 2 7.10 -> 6.69, EED sigma 2 6.64 -> 5.93)
    HaloItems<H::K> items;
    halo_items<G::SU_W, H, G::NTHR>(items, w, h, pitch, x0, y0, we, he);
    int m = 0, k = 0;  // cycle of this launch, step of the cycle
    for (;;) {
        const bool last = k == a.n - 1;
        const bool end = last && m == a.cycles - 1;
        const float alpha = a.alpha[k], alpha_lo = a.alpha_lo[k];
        const float *const c0 = a.u[m & 1];
        float *const c1 = a.u[(m + 1) & 1];
        ++tag;
        unsigned long long *const halo = a.halo + (tag & 1) * (long)h * pitch;
        tile_tensor<R, EED, TH, VAR, LAT>(p, p.c4, su, sx, ss);
        __syncthreads();
        float nu[ER][4];
        double rnum = 0.0, rden = 0.0;
        tile_divergence<R, EED, TH, LAT>(su, sx, w, h, x0, y0, [&](const int e, const int gy, const int gx,
                                                                   const float *ucv, const float *Pu) {
            fsi_update4<U>(prev[e], ucv, Pu, mk[e], alpha, alpha_lo, p.tau_t, p.tau_lo, nu[e]);
            const long gi = (long)gy * pitch + gx;
            const bool full = gx + 3 < w;
            const int r = re + e;
            if (r < H::HL || r >= he - H::HL || 4 * qe < H::HE || 4 * qe + 3 >= we - H::HE) {
                if (full) {
                    halo_store2(halo + gi, nu[e][0], nu[e][1], tag);
                    halo_store2(halo + gi + 2, nu[e][2], nu[e][3], tag);
                } else {
                    for (int j = 0; j < 4; ++j)
                        if (gx + j < w) halo_store(halo + gi + j, nu[e][j], tag);
                }
            }
            if (!EED) {  // this thread alone reads these pixels in stage E
                float *d = su + (r + G::HL) * G::SU_W + 4 * qe + 8;
                if (full) {
                    *reinterpret_cast<float4 *>(d) = make_float4(nu[e][0], nu[e][1], nu[e][2], nu[e][3]);
                } else {
                    for (int j = 0; j < 4; ++j)
                        if (gx + j < w) d[j] = nu[e][j];
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) prev[e][j] = last ? nu[e][j] : ucv[j];  // u^{m+1,-1} = u^{m+1,0}
            if (last) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (gx + j < w) {
                        const double d = double(nu[e][j]) - double(c0[gi + j]);
                        rnum += d * d;
                        rden += double(nu[e][j]) * double(nu[e][j]);
                    }
                if (full) {
                    *reinterpret_cast<float4 *>(c1 + gi) = make_float4(nu[e][0], nu[e][1], nu[e][2], nu[e][3]);
                } else {
                    for (int j = 0; j < 4; ++j)
                        if (gx + j < w) c1[gi + j] = nu[e][j];
                }
            }
        });
        if (last) {
            if (m > 0 && !cycle_goes_on(p.ctl, cycle0 + m, &s_dead, a.poll0)) break;  // cycle m - 1 was the last one
            cycle_change(rnum, rden, p.ctl, p.partials, ntiles, bid, cycle0 + m + 1, red);
            ++m;
        }
        if (end) break;
        k = last ? 0 : k + 1;
        if (EED) {  // stage E reads the neighbours' pixels of the window: write once all have
            __syncthreads();
#pragma unroll
            for (int e = 0; e < ER; ++e)
                if (re + e < TH && y0 + re + e < h)
                    for (int j = 0; j < 4; ++j)
                        if (x0 + 4 * qe + j < w) su[(re + e + G::HL) * G::SU_W + 4 * qe + 8 + j] = nu[e][j];
        }
        if (!gather_halo(items, halo, tag, su, p.ctl, a.poll0)) {
            s_dead = 1;
            *(volatile int *)&p.ctl->timeout = 1;
        }
        __syncthreads();
        if (s_dead) break;
    }
    // m cycles of this launch count; their last iterate is in u[m & 1]
    if (m & 1) {
#pragma unroll
        for (int e = 0; e < ER; ++e)
            for (int j = 0; j < 4; ++j)
                if (re + e < TH && y0 + re + e < h && x0 + 4 * qe + j < w) {
                    const long gi = (long)(y0 + re + e) * pitch + x0 + 4 * qe + j;
                    a.u[0][gi] = a.u[1][gi];
                }
    }
}

// Sets the attributes of a cooperative kernel; *room: how many of its CTAs fit the current
// device at once.
template <typename Kern>
cudaError_t cycle_room(Kern kern, int threads, size_t smem, int *room)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int per_sm = 0, dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    *room = per_sm * sms;
    return e;
}

template <typename Kern, typename Args>
cudaError_t cycle_cooperative(Kern kern, dim3 grid, int threads, size_t smem, cudaStream_t s, const Args &a)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// Launches the cycles; with a == nullptr prepares the kernel (cycle_room).
template <int R, bool EED, typename U, int TH, int LAT, bool VAR>
cudaError_t launch_fsi_cycle(const CycleArgs *ap, int *room, cudaStream_t s)
{
    using G = FastTile<R, EED, TH, LAT>;
    auto kern = fsi_cycle_fast<R, EED, U, TH, LAT, VAR>;
    if (!ap) return cycle_room(kern, G::NTHR, G::SMEM, room);
    return cycle_cooperative(kern, dim3((ap->s.w + 63) / 64, (ap->s.h + TH - 1) / TH), G::NTHR, G::SMEM, s, *ap);
}

template <bool EED, typename U, int TH, int LAT, bool VAR>
cudaError_t cycle_radius(const CycleArgs *a, int R, int *room, cudaStream_t s)
{
    switch (R) {
    case 0: return launch_fsi_cycle<0, EED, U, TH, LAT, VAR>(a, room, s);
    case 1: return launch_fsi_cycle<1, EED, U, TH, LAT, VAR>(a, room, s);
    case 2: return launch_fsi_cycle<2, EED, U, TH, LAT, VAR>(a, room, s);
    case 3: return launch_fsi_cycle<3, EED, U, TH, LAT, VAR>(a, room, s);
    case 4: return launch_fsi_cycle<4, EED, U, TH, LAT, VAR>(a, room, s);
    case 5: return launch_fsi_cycle<5, EED, U, TH, LAT, VAR>(a, room, s);
    case 6: return launch_fsi_cycle<6, EED, U, TH, LAT, VAR>(a, room, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace foeed
