// FSI cycles of a small FP64 image in one cooperative launch: cycle_fast.cuh with the stages
// of step_kernel.cuh. A halo pixel travels as two (half, tag) words; both carry the tag, so
// a pixel is taken when both are the step's. One thread per output pixel. A tile may be lower
// than the halo: it then gathers from two tiles above and below, and all of its pixels are
// published. That a word is overwritten two steps later only holds as there: a tile that
// needs a pixel of another, directly or mirrored, is within the halo of it, and so the
// other way round.
//
// Bound: the FP64 pipe, two operations a cycle and SM (64 x 64 on 8 x 4 tiles: 1.3 of the 4.0 us;
// 256 x 256 on 16 x 16: 12.4 of 16.5), then the exchange. us a step, FOEED, sigma 1, one launch
// per step -> this: 16 x 16 5.28 -> 4.05, 64 x 64 5.15 -> 4.03 (8 x 4 tiles; 4.40 on 8 x 8, 9.78
// on 16 x 16), 128 x 128 8.16 -> 6.52 (8 x 8; 7.19 on 8 x 4), 192 x 192 11.50 -> 9.79 (16 x 16),
// 256 x 256 18.24 -> 16.47; EED 64 x 64 4.62 -> 3.47; sigma 2 64 x 64
// 6.26 -> 4.93. With four 16 x 16 tiles per SM (340 x 340, EED) 25.27 -> 26.28: left to the step
// kernels.
#pragma once

#include <algorithm>

#include "cycle_fast.cuh"
#include "step_kernel.cuh"

namespace foeed {

template <int R, int TW, int TH, bool EED>
__global__ void __launch_bounds__(kThreads) fsi_cycle_f64(const __grid_constant__ CycleArgs64 a)
{
    using G = Tile<R, TW, TH, EED>;
    static_assert(TW * TH <= kThreads, "one output pixel per thread");
    constexpr int NI = G::SU_W * G::SU_H, K = (NI + kThreads - 1) / kThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *const su = reinterpret_cast<double *>(smem_raw);
    __shared__ double red[64];
    __shared__ int s_dead;
    const StepArgs<double> &p = a.s;
    if (p.ctl->done) return;
    const int tid = threadIdx.x, w = p.w, h = p.h, pitch = (int)p.pitch;
    const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH;
    const int we = min(TW, w - x0), he = min(TH, h - y0);
    const int ntiles = gridDim.x * gridDim.y, bid = blockIdx.y * gridDim.x + blockIdx.x;
    const int cycle0 = p.ctl->cycles;
    uint32_t tag = (uint32_t)cycle0 * (uint32_t)a.n;
    if (tid == 0) s_dead = 0;
    // the window, and the pixels of it this thread gathers from then on: those of other tiles
    // and the mirrored ones (negative: none)
    int from[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const int i = tid + j * kThreads, r = i / G::SU_W, c = i - r * G::SU_W;
        from[j] = -1;
        if (i < NI && r < he + 2 * G::HL && c < we + 2 * G::HL) {
            const int o = reflect(y0 - G::HL + r, h) * pitch + reflect(x0 - G::HL + c, w);
            su[i] = a.u[0][o];
            if (r < G::HL || r >= he + G::HL || c < G::HL || c >= we + G::HL) from[j] = o;
        }
    }
    const int px = tid % TW, py = tid / TW;
    const bool own = py < he && px < we;
    const bool seen = px < G::HL || px >= we - G::HL || py < G::HL || py >= he - G::HL;  // another tile or a mirror needs it
    const int gi = (y0 + py) * pitch + x0 + px;
    const bool known = own && p.mask[gi] != 0;
    double prev = own ? a.u[0][gi] : 0.0;
    __syncthreads();
    int m = 0, k = 0;  // cycle of this launch, step of the cycle
    for (;;) {
        const bool last = k == a.n - 1;
        const bool end = last && m == a.cycles - 1;
        ++tag;
        unsigned long long *const halo = a.halo + (tag & 1) * 2l * h * pitch;
        general_tensor<double, R, TW, TH, EED>(p, su);
        __syncthreads();
        double un = 0.0, rnum = 0.0, rden = 0.0;
        if (own) {
            double uc;
            const double Pu = general_divergence<double, R, TW, TH, EED>(su, px, py, uc);
            const double ex = uc - p.tau_t * Pu;
            un = known ? uc : prev + a.alpha[k] * (ex - prev);
            if (seen) {
                const unsigned long long t = (unsigned long long)tag << 32;
                asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(halo + 2l * gi),
                             "l"(t | (uint32_t)__double2hiint(un)), "l"(t | (uint32_t)__double2loint(un))
                             : "memory");
            }
            prev = last ? un : uc;
            if (last) {
                const double d = un - a.u[m & 1][gi];
                rnum = d * d;
                rden = un * un;
                a.u[(m + 1) & 1][gi] = un;
            }
        }
        if (last) {
            if (m > 0 && !cycle_goes_on(p.ctl, cycle0 + m, &s_dead, a.poll0)) break;
            cycle_change(rnum, rden, p.ctl, p.partials, ntiles, bid, cycle0 + m + 1, red);
            ++m;
        }
        if (end) break;
        k = last ? 0 : k + 1;
        if (EED) __syncthreads();  // the divergence reads the neighbours' pixels of the window
        if (own) su[(py + G::HL) * G::SU_W + px + G::HL] = un;
        uint32_t pend = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) pend |= from[j] >= 0 ? 1u << j : 0u;
        for (int it = a.poll0; pend; ++it) {
            unsigned long long hi[K], lo[K];
#pragma unroll
            for (int j = 0; j < K; ++j)
                if (pend >> j & 1) halo_load2(halo + 2l * from[j], hi[j], lo[j]);
#pragma unroll
            for (int j = 0; j < K; ++j)
                if ((pend >> j & 1) && (uint32_t)(hi[j] >> 32) == tag && (uint32_t)(lo[j] >> 32) == tag) {
                    su[tid + j * kThreads] = __hiloint2double((int)(uint32_t)hi[j], (int)(uint32_t)lo[j]);
                    pend &= ~(1u << j);
                }
            if ((it & 1023) == 1023 && (it >= kPollLimit || *(volatile const int *)&p.ctl->timeout)) {
                s_dead = 1;
                *(volatile int *)&p.ctl->timeout = 1;
                break;
            }
        }
        __syncthreads();
        if (s_dead) break;
    }
    if ((m & 1) && own) a.u[0][gi] = a.u[1][gi];
}

template <int R, int TW, int TH, bool EED>
cudaError_t launch_cycle_f64(const CycleArgs64 *ap, int *room, cudaStream_t s)
{
    constexpr size_t smem = sizeof(double) * Tile<R, TW, TH, EED>::ELEMS;
    auto kern = fsi_cycle_f64<R, TW, TH, EED>;
    if (!ap) return cycle_room(kern, kThreads, smem, room);
    return cycle_cooperative(kern, dim3((ap->s.w + TW - 1) / TW, (ap->s.h + TH - 1) / TH), kThreads, smem, s, *ap);
}

// The tile shape (4: 8 x 4, 8: 8 x 8, 16: 16 x 16, 0: the step kernels) of a w x h image: the
// one whose busiest SM has the fewest FP64 operations, if that is no more than the step
// kernels' wide shapes have and what a launch costs beside a halo exchange (2 us of them).
// (300 x 300: 25.8 us a step here, 21.8 on 32 x 20 tiles. Against the narrow shapes, whose
// tiles take longer than their operations say, it always pays: 200 x 200 16.8, steps on 8 x 8
// 17.3; sigma 2 20.4, 22.3.)
template <int R, bool EED>
int cycle_shape_f64(const int w, const int h)
{
    auto count = [&](int tw, int th) { return (long)((w + tw - 1) / tw) * ((h + th - 1) / th); };
    auto cost = [&](int tw, int th, long ops) { return (count(tw, th) + kSMs - 1) / kSMs * ops; };
    // reduction partials the workspace holds (max_blocks in api.cu), two sets of them
    const long room = std::max(count(kTileW64, kTileH64), (long)kPartialsMin) / 2;
    long step = 0;
    f64_step_shape<R, EED>(w, h, false, &step);
    int best = 0;
    long least = step + 8000;
    auto consider = [&](int shape, int tw, int th, long ops) {
        const long c = cost(tw, th, ops);
        if (count(tw, th) <= room && c <= least) { best = shape; least = c; }
    };
    consider(4, 8, 4, f64_tile_ops<R, 8, 4, EED>());
    consider(16, 16, 16, f64_tile_ops<R, 16, 16, EED>());
    consider(8, 8, 8, f64_tile_ops<R, 8, 8, EED>());
    return best;
}

// With a == nullptr: *shape and *room of a w x h image; else launches shape *shape.
template <bool EED>
cudaError_t cycle_f64(const CycleArgs64 *a, int R, int w, int h, int *shape, int *room, cudaStream_t s)
{
    switch (R) {
#define CYCLE_R(r)                                                                                        \
    case r:                                                                                               \
        if (!a) *shape = cycle_shape_f64<r, EED>(w, h);                                                   \
        return *shape == 4    ? launch_cycle_f64<r, 8, 4, EED>(a, room, s)                                \
               : *shape == 8  ? launch_cycle_f64<r, 8, 8, EED>(a, room, s)                                \
               : *shape == 16 ? launch_cycle_f64<r, 16, 16, EED>(a, room, s)                              \
                              : cudaSuccess;
    CYCLE_R(0) CYCLE_R(1) CYCLE_R(2) CYCLE_R(3) CYCLE_R(4) CYCLE_R(5) CYCLE_R(6)
#undef CYCLE_R
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace foeed
