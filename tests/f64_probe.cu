// Test access to two parts of the FP64 step: the tile its size rule takes (host code) and the
// reciprocal and roots of its tensor stage.
#include "step_kernel.cuh"

template <int R>
static int shape(const bool eed, const int w, const int h)
{
    long cost = 0;
    return eed ? foeed::f64_step_shape<R, true>(w, h, true, &cost) : foeed::f64_step_shape<R, false>(w, h, true, &cost);
}

// tile width * 100 + height
extern "C" int f64_probe_tile(const int R, const int eed, const int w, const int h)
{
    static const int tile[8] = {3232, 3216, 1616, 808, 804, 3228, 3224, 3220};
    switch (R) {
    case 0: return tile[shape<0>(eed, w, h)];
    case 1: return tile[shape<1>(eed, w, h)];
    case 2: return tile[shape<2>(eed, w, h)];
    case 3: return tile[shape<3>(eed, w, h)];
    case 4: return tile[shape<4>(eed, w, h)];
    case 5: return tile[shape<5>(eed, w, h)];
    case 6: return tile[shape<6>(eed, w, h)];
    default: return 0;
    }
}

static __global__ void roots(const double *x, double *out, const int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        out[i] = foeed::f64_rcp(x[i]);
        out[n + i] = foeed::f64_rsqrt(x[i]);
        out[2 * n + i] = foeed::f64_rsqrt4(x[i]);
    }
}

// x (n) and out (3 n: 1/x, x^-1/2, x^-1/4): device pointers
extern "C" int f64_probe_roots(const double *x, double *out, const int n)
{
    roots<<<64, 256>>>(x, out, n);
    return (int)cudaDeviceSynchronize();
}
