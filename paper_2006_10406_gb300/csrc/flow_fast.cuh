// FSI cycles of a larger image in one cooperative launch: the CTAs that fit the GPU take
// (step, tile) pairs in order from one counter, so that the tail of a step runs beside the
// head of the next one.
//
// A tile of step k + 1 needs itself and its eight neighbours to have finished step k: for
// their pixels, and because it writes where they read. Each tile counts the steps it has
// finished in done[tile] (release after its stores, acquire before the window load). Pairs
// are handed out in order, so the tiles a pair waits for are running or finished; in an
// image of more tiles than CTAs they finished long ago. A cycle's change is summed by the
// last tile of its last step (cycle_change); pairs of the next cycle wait for the verdict.
// What other CTAs wrote is read through the L2 (cp.async.cg, ld.cg). Waits are bounded, as
// in cycle_fast.cuh.
//
// Saves the launch, fill and drain of every step (5.7 us of a 2048 x 2048 step's 25.8);
// costs two barriers, the flags and 11% more warp instructions (what a CTA works out once is
// worked out per tile, and the tensor stage spills a little at 64 registers).
// us a step, FOEED (EED), sigma 1.5, 20 cycles of 40 steps, one launch per step -> this: 1536 x
// 1536 16.7 -> 14.1 (17.3 -> 14.7), 1080 x 1920 15.2 -> 12.9 (15.6 -> 13.4), 2048 x 2048 25.8 ->
// 23.6 (27.1 -> 24.7), 2560 x 2560 37.6 -> 36.5 (39.8 -> 38.2); 2160 x 3840 even, 4096 x 4096
// 91.6 -> 96.2. Short cycles and launches: use_flow in api.cu.
// 64 x 16 tiles cost more instructions a pixel but let 0.8 to 1.4 megapixels overlap steps; one
// launch per step (from 1100 x 1100: this on 64 x 32 tiles) -> 64 x 16 tiles, FOEED sigma 1, sigma 2
// and EED sigma 2: 704 x 1100 8.12 -> 8.39, 8.63 -> 8.92, 8.65 -> 8.98 (left to the step kernels);
// 720 x 1280 8.88 -> 8.15, 9.63 -> 8.88, 9.94 -> 9.03; 1000 x 1024 9.61 -> 8.26, 10.53 -> 9.16,
// 10.78 -> 9.33; 1100 x 1100 10.81 -> 9.44, 11.47 -> 10.51, 11.64 -> 10.67; 1000 x 1400 10.94 ->
// 10.32, 11.74 -> 11.46, 12.02 -> 11.69; 1200 x 1400 11.42 -> 12.17 (left to 64 x 32 tiles). With
// the two-float update, sigma 2: 640 x 1024 9.33 -> 9.01, 630 x 1030 9.36 -> 9.35, 704 x 1100
// 9.34 -> 9.23, 1000 x 1024 11.32 -> 9.65. A step cannot take less than its tile's chain of flags,
// window, stages and store, some 8 us with four tiles per SM. Up to 608 tiles of 64 x 24 the
// resident-tile kernel goes first where it is faster (kCycleKinds in api.cu).
#pragma once

#include "cycle_fast.cuh"

namespace foeed {

// Whether the pair (step, tile) may start: need = steps its neighbourhood must have
// finished; verdict of cycle number `cycle` (0: none) must be known and to go on. Called by
// one warp; false if the solve ended or a wait ran out.
__device__ __forceinline__ bool flow_ready(const FlowArgs &a, const int ntx, const int nty, const int tx, const int ty,
                                           const int need, const int cycle)
{
    const int lane = threadIdx.x & 31;
    Ctl *ctl = a.s.ctl;
    const int nx = tx + lane % 3 - 1, ny = ty + lane / 3 - 1;
    const bool flag = lane < 9 && nx >= 0 && nx < ntx && ny >= 0 && ny < nty;
    const int *src = flag ? a.done + ny * ntx + nx : &ctl->verdict[cycle & 1];
    bool ok = true, wait = flag || (lane == 9 && cycle > 0);
    for (int it = a.poll0; wait; ++it) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(src) : "memory");
        wait = flag ? v < need : v != cycle && v != -cycle;
        ok = flag || v != -cycle;
        if (wait && (it & 15) == 15 &&
            (it >= kPollLimit || *(volatile const int *)&ctl->timeout || *(volatile const int *)&ctl->done)) {
            if (it >= kPollLimit) *(volatile int *)&ctl->timeout = 1;
            wait = ok = false;
        }
    }
    return __all_sync(0xffffffffu, ok);
}

template <int R, bool EED, typename U, int TH, int LAT>
__global__ void __launch_bounds__(256, 4) fsi_flow_fast(const __grid_constant__ FlowArgs a)
{
    using G = FastTile<R, EED, TH, LAT>;
    constexpr int ER = G::ER;
    extern __shared__ __align__(16) float sm[];
    __shared__ double red[64];
    __shared__ int s_pair[5];  // cycle of this launch (negative: none left), step, tile column and row; ready
    const StepArgs<float> &p = a.s;
    float *su = sm, *sx = su + G::SU_W * G::SU_H, *ss = sx + G::SXT;
    const int tid = threadIdx.x, w = p.w, h = p.h;
    const long pitch = p.pitch;
    const int ntx = (w + 63) / 64, nty = (h + TH - 1) / TH, ntiles = ntx * nty;
    const int cycle0 = (int)a.ticket[1];  // as an argument, 2048 x 2048 takes 1% longer
    auto decode = [&](const unsigned int t) {
        const int step = (int)(t / (unsigned)ntiles), tile = (int)(t - (unsigned)step * ntiles);
        const int c = step / a.n;
        s_pair[0] = c < a.cycles ? c : -1;
        s_pair[1] = step - c * a.n;
        s_pair[3] = tile / ntx;
        s_pair[2] = tile - s_pair[3] * ntx;
    };
    // warp 0 hands out pairs, warp 1 stores the flags. A CTA may start after others have ended
    // cycles, so what they store in the control block is looked at by one thread only, and the
    // launch's first cycle is the host's word.
    if (tid == 0) {
        if (*(volatile const int *)&p.ctl->done || *(volatile const int *)&p.ctl->timeout)
            s_pair[0] = -1;
        else
            decode(atomicAdd(a.ticket, 1u));
    }
    __syncthreads();
    for (;;) {
        const int c = s_pair[0], k = s_pair[1], tx = s_pair[2], ty = s_pair[3];
        if (c < 0) break;
        const int steps = (cycle0 + c) * a.n + k;  // of the solve, before this one
        if (tid < 32) {
            const bool ok = flow_ready(a, ntx, nty, tx, ty, steps, c > 0 ? cycle0 + c : 0);
            if (tid == 0) s_pair[4] = ok;
        }
        __syncthreads();
        if (!s_pair[4]) break;
        unsigned int next = 0;
        if (tid == 0) next = atomicAdd(a.ticket, 1u);
        const bool last = k == a.n - 1;
        const float *const uprev = k < 2 ? a.C : (k & 1 ? a.B : a.A);
        const float *const ucur = k == 0 ? a.C : (k & 1 ? a.A : a.B);
        float *const unext = last ? a.C : (k & 1 ? a.B : a.A);
        const int x0 = tx * 64, y0 = ty * TH;
        tile_window<R, EED, TH, LAT, true>(ucur, w, h, pitch, x0, y0, su);
        tile_window_wait();
        tile_tensor<R, EED, TH, false, LAT>(p, p.c4, su, sx, ss);
        const int qe = tid % 16, re = ER * (tid / 16);
        float4 pre_up[ER];
        uint32_t pre_mk[ER];
#pragma unroll
        for (int e = 0; e < ER; ++e) {
            const int gy = y0 + re + e, gx = x0 + 4 * qe;
            pre_up[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            pre_mk[e] = 0u;
            if (gy < h && gx < w) {  // the internal pitch is a multiple of 32: whole groups lie inside the rows
                pre_up[e] = __ldcg(reinterpret_cast<const float4 *>(uprev + (long)gy * pitch + gx));
                pre_mk[e] = __ldg(reinterpret_cast<const unsigned int *>(p.mask + (long)gy * pitch + gx));
            }
        }
        __syncthreads();
        double rnum = 0.0, rden = 0.0;
        tile_divergence<R, EED, TH, LAT>(su, sx, w, h, x0, y0, [&](const int e, const int gy, const int gx, const float *ucv,
                                                              const float *Pu) {
            const long gi = (long)gy * pitch + gx;
            const float upv[4] = {pre_up[e].x, pre_up[e].y, pre_up[e].z, pre_up[e].w};
            float un[4];
            fsi_update4<U>(upv, ucv, Pu, pre_mk[e], a.alpha[k], a.alpha_lo[k], p.tau_t, p.tau_lo, un);
            if (last) {
                const float4 c4 = __ldcg(reinterpret_cast<const float4 *>(a.C + gi));
                const float c0v[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (gx + j < w) {
                        const double d = double(un[j]) - double(c0v[j]);
                        rnum += d * d;
                        rden += double(un[j]) * double(un[j]);
                    }
            }
            if (gx + 3 < w) {
                *reinterpret_cast<float4 *>(unext + gi) = make_float4(un[0], un[1], un[2], un[3]);
            } else {
                for (int j = 0; j < 4; ++j)
                    if (gx + j < w) unext[gi + j] = un[j];
            }
        });
        if (last) cycle_change(rnum, rden, p.ctl, p.partials, ntiles, ty * ntx + tx, cycle0 + c + 1, red);
        if (tid == 0) decode(next);
        __syncthreads();
        if (tid == 32)
            asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.done + ty * ntx + tx), "r"(steps + 1) : "memory");
    }
}

// Launches the cycles; with a == nullptr sets the kernel's attributes and reports in *room
// how many of its CTAs fit the current device at once.
template <int R, bool EED, typename U, int TH, int LAT>
cudaError_t launch_fsi_flow(const FlowArgs *ap, int *room, cudaStream_t s)
{
    using G = FastTile<R, EED, TH, LAT>;
    auto kern = fsi_flow_fast<R, EED, U, TH, LAT>;
    if (!ap) return cycle_room(kern, 256, G::SMEM, room);
    return cycle_cooperative(kern, dim3(*room), 256, G::SMEM, s, *ap);
}

template <bool EED, int TH, int LAT>
cudaError_t flow_radius(const FlowArgs *a, bool f64_update, int R, int *room, cudaStream_t s)
{
    switch (R) {
#define FLOW_R(r)                                                              \
    case r:                                                                    \
        return f64_update ? launch_fsi_flow<r, EED, double, TH, LAT>(a, room, s) \
                          : launch_fsi_flow<r, EED, float, TH, LAT>(a, room, s);
    FLOW_R(0) FLOW_R(1) FLOW_R(2) FLOW_R(3) FLOW_R(4) FLOW_R(5) FLOW_R(6)
#undef FLOW_R
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace foeed
