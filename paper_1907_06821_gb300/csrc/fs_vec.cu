// Band-wise vector kernels of the solver: residual norms and inner products
// (warp-shuffle + shared-memory tree, a cluster of blocks per band, fixed order so
// that repeated runs give identical bits), the preconditioned residual, row
// normalisation, start-block generation and precision conversion.
//
// The sums are FP64 also in the FP32 stage, so the FP64 units bound them (2 operations a
// clock and SM): a band is spread over a cluster of up to 8 blocks whose partial sums meet in
// distributed shared memory, and float values are widened with integer instructions (the
// conversion runs on the FP64 units as well).  36 bands of 41,657 plane waves, with one block a
// band, left three quarters of the SMs idle: 0.1 ms a call.
#include "fs_common.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace cg = cooperative_groups;

namespace {

constexpr int RT = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// sum over the block; every thread gets the result
__device__ double block_sum(double v, double* sh) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double t = 0;
    const int nw = blockDim.x >> 5;
    if (wid == 0) {
        t = lane < nw ? sh[lane] : 0.0;
        t = warp_sum(t);
        if (lane == 0) sh[32] = t;
    }
    __syncthreads();
    return sh[32];
}

// exact widening; floats below 2^-126 read as zero
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(float x) {
    const uint32_t u = __float_as_uint(x), e = (u >> 23) & 255;
    if (e == 255) return (double)x;  // Inf, NaN
    const uint32_t hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20));
    return e ? __hiloint2double((int)hi, (int)(u << 29)) : 0.0;
}
template <typename T2> __device__ __forceinline__ double2 wide2(T2 v) { return make_double2(wide(v.x), wide(v.y)); }

// sum over the cluster of NV values per thread; every thread gets the totals.  slot: shared
// array of 2 NV doubles, used in turn (turn counts the calls of a kernel)
template <int NV>
__device__ __forceinline__ void cluster_sum(double (&v)[NV], double* sh, double* slot, int& turn) {
    cg::cluster_group cl = cg::this_cluster();
    double* mine = slot + (turn & 1) * NV;
    ++turn;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const double t = block_sum(v[i], sh);
        if (threadIdx.x == 0) mine[i] = t;
    }
    cl.sync();
    const int n = (int)cl.num_blocks();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        double t = 0;
        for (int r = 0; r < n; ++r) t += *cl.map_shared_rank(mine + i, r);
        v[i] = t;
    }
}

// this block's share [g0, g1) of a band
__device__ __forceinline__ void share(long npw, long& g0, long& g1) {
    const int n = (int)cg::this_cluster().num_blocks(), r = (int)cg::this_cluster().block_rank();
    const long per = (npw + n - 1) / n;
    g0 = min(npw, r * per);
    g1 = min(npw, g0 + per);
}

// dot = <x, y>, resid = || y - dot x ||; RH (optional) = y - dot x, the H residual
template <typename T2>
__global__ void __launch_bounds__(RT) resid_kernel(const T2* __restrict__ X, const T2* __restrict__ Y, long npw,
                                                   double* resid, double2* dot, T2* RH) {
    using Rl = typename real_of<T2>::t;
    __shared__ double sh[33], slot[4];
    int turn = 0;
    const long band = blockIdx.y;
    const T2* x = X + band * npw;
    const T2* y = Y + band * npw;
    long g0, g1;
    share(npw, g0, g1);
    double d[2] = {0, 0};
    for (long g = g0 + threadIdx.x; g < g1; g += RT) {
        const double2 a = wide2(x[g]), b = wide2(y[g]);
        d[0] = fma(a.x, b.x, fma(a.y, b.y, d[0]));
        d[1] = fma(a.x, b.y, fma(-a.y, b.x, d[1]));
    }
    cluster_sum<2>(d, sh, slot, turn);
    double s[1] = {0};
    for (long g = g0 + threadIdx.x; g < g1; g += RT) {
        const double2 a = wide2(x[g]), b = wide2(y[g]);
        const double rx = fma(-d[0], a.x, fma(d[1], a.y, b.x));
        const double ry = fma(-d[0], a.y, fma(-d[1], a.x, b.y));
        s[0] = fma(rx, rx, fma(ry, ry, s[0]));
        if (RH) RH[band * npw + g] = mk((Rl)rx, (Rl)ry);
    }
    __shared__ double slot1[2];
    turn = 0;
    cluster_sum<1>(s, sh, slot1, turn);
    if (threadIdx.x == 0 && cg::this_cluster().block_rank() == 0) {
        resid[band] = sqrt(s[0]);
        if (dot) dot[band] = make_double2(d[0], d[1]);
    }
    cg::this_cluster().sync();  // nobody leaves while its sums are read
}

// resid = || y - shift_i x ||
template <typename T2>
__global__ void __launch_bounds__(RT) resid_shift_kernel(const T2* __restrict__ X, const T2* __restrict__ Y,
                                                         const double* __restrict__ shift, long npw, double* resid) {
    __shared__ double sh[33], slot[2];
    int turn = 0;
    const long band = blockIdx.y;
    const T2* x = X + band * npw;
    const T2* y = Y + band * npw;
    const double s0 = shift[band];
    long g0, g1;
    share(npw, g0, g1);
    double s[1] = {0};
    for (long g = g0 + threadIdx.x; g < g1; g += RT) {
        const double2 a = wide2(x[g]), b = wide2(y[g]);
        const double rx = fma(-s0, a.x, b.x), ry = fma(-s0, a.y, b.y);
        s[0] = fma(rx, rx, fma(ry, ry, s[0]));
    }
    cluster_sum<1>(s, sh, slot, turn);
    if (threadIdx.x == 0 && cg::this_cluster().block_rank() == 0) resid[band] = sqrt(s[0]);
    cg::this_cluster().sync();
}

// rows of X (and of Y, when given) divided by the norm of X's row
template <typename T2>
__global__ void __launch_bounds__(RT) normalize_kernel(T2* X, T2* Y, const int* __restrict__ map, long npw) {
    using R = typename real_of<T2>::t;
    __shared__ double sh[33], slot[2];
    int turn = 0;
    const long row = map ? map[blockIdx.y] : blockIdx.y;
    T2* x = X + row * npw;
    T2* y = Y ? Y + row * npw : nullptr;
    long g0, g1;
    share(npw, g0, g1);
    double s[1] = {0};
    for (long g = g0 + threadIdx.x; g < g1; g += RT) {
        const double2 a = wide2(x[g]);
        s[0] = fma(a.x, a.x, fma(a.y, a.y, s[0]));
    }
    cluster_sum<1>(s, sh, slot, turn);
    const double f = sqrt(s[0]);
    const R inv = (R)(f > 0 ? 1.0 / f : 0.0);
    for (long g = g0 + threadIdx.x; g < g1; g += RT) {
        x[g] = cscale(x[g], inv);
        if (y) y[g] = cscale(y[g], inv);
    }
    cg::this_cluster().sync();
}

// kinetic energy of each band: sum_g |q_g|^2/2 |x_g|^2 / sum_g |x_g|^2
template <typename T2>
__global__ void __launch_bounds__(RT) band_kin_kernel(const T2* __restrict__ X, const double* __restrict__ kin, long npw,
                                                      double* out) {
    __shared__ double sh[33];
    const T2* x = X + (long)blockIdx.x * npw;
    double s = 0, n = 0;
    for (long g = threadIdx.x; g < npw; g += blockDim.x) {
        T2 a = x[g];
        double p = (double)a.x * a.x + (double)a.y * a.y;
        s += kin[g] * p;
        n += p;
    }
    s = block_sum(s, sh);
    n = block_sum(n, sh);
    if (threadIdx.x == 0) out[blockIdx.x] = n > 0 ? s / n : 0.0;
}

// W[a] = M_i(q) R[act[a]]
//   precond 0: paper's M(q) = 1 / ((|q|^2/2 - E)^2 + dE^2)
//   precond 1: folded Teter-Payne-Allan form K(x)^2 / T_i^2 with x = (|q|^2/2) / T_i
template <typename T2>
__global__ void make_w_kernel(const T2* __restrict__ R, const int* __restrict__ act, long npw, T2* __restrict__ W,
                              const double* __restrict__ kin, double e_ref, double dE2, int precond,
                              const double* __restrict__ band_kin) {
    using Rl = typename real_of<T2>::t;
    const int i = act[blockIdx.y];
    const T2* r = R + (long)i * npw;
    T2* w = W + (long)blockIdx.y * npw;
    double tk = band_kin ? fmax(band_kin[i], 1e-3) : 1.0;
    for (long g = blockIdx.x * (long)blockDim.x + threadIdx.x; g < npw; g += (long)gridDim.x * blockDim.x) {
        double m;
        if (precond == 1) {
            double xx = kin[g] / tk;
            double num = 27.0 + xx * (18.0 + xx * (12.0 + 8.0 * xx));
            double kk = num / (num + 16.0 * xx * xx * xx * xx);
            m = kk * kk / (tk * tk);
        } else if (precond == 2) {  // lowest states of H itself: 1 / (1 + |q|^2 / 2)
            m = 1.0 / (1.0 + kin[g]);
        } else {
            double d = kin[g] - e_ref;
            m = 1.0 / (d * d + dE2);
        }
        T2 a = r[g];
        w[g] = mk((Rl)m * a.x, (Rl)m * a.y);
    }
}

// A residual from the H residual r = y - d x:  (H-E)^2 x - theta x
//   = (H-E) r + d r + (d^2 - theta) x,   written over RH;  ra_i = its norm.
// Every term is computed from the small vector r, so its rounding error
// scales with ||r|| instead of with ||(H-E) y||.
template <typename T2>
__global__ void __launch_bounds__(RT) a_resid_kernel(const T2* __restrict__ ZR, T2* RH, const T2* __restrict__ X,
                                                     const double2* __restrict__ dots,
                                                     const double* __restrict__ theta, long npw, double* ra) {
    using Rl = typename real_of<T2>::t;
    __shared__ double sh[33], slot[2];
    int turn = 0;
    const long i = blockIdx.y;
    const double2 d = dots[i];
    const double c0x = d.x * d.x - d.y * d.y - theta[i], c0y = 2.0 * d.x * d.y;
    const T2* z = ZR + i * npw;
    const T2* x = X + i * npw;
    T2* r = RH + i * npw;
    long g0, g1;
    share(npw, g0, g1);
    double s[1] = {0};
    for (long g = g0 + threadIdx.x; g < g1; g += RT) {
        const double2 a = wide2(z[g]), b = wide2(r[g]), c = wide2(x[g]);
        const double ox = fma(d.x, b.x, fma(-d.y, b.y, a.x)) + fma(c0x, c.x, -c0y * c.y);
        const double oy = fma(d.x, b.y, fma(d.y, b.x, a.y)) + fma(c0x, c.y, c0y * c.x);
        r[g] = mk((Rl)ox, (Rl)oy);
        s[0] = fma(ox, ox, fma(oy, oy, s[0]));
    }
    cluster_sum<1>(s, sh, slot, turn);
    if (threadIdx.x == 0 && cg::this_cluster().block_rank() == 0) ra[i] = sqrt(s[0]);
    cg::this_cluster().sync();
}

// splitmix64 (Steele, Lea and Flood 2014) as a counter-based generator
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

__global__ void damp_random_kernel(double2* X, long npw, int first, unsigned long long seed,
                                   const double* __restrict__ kin) {
    const long band = first + blockIdx.y;
    for (long g = blockIdx.x * (long)blockDim.x + threadIdx.x; g < npw; g += (long)gridDim.x * blockDim.x) {
        unsigned long long ctr = ((unsigned long long)band << 32) ^ (unsigned long long)g;
        unsigned long long h1 = splitmix64(seed ^ splitmix64(2 * ctr));
        unsigned long long h2 = splitmix64(seed ^ splitmix64(2 * ctr + 1));
        double u1 = ((h1 >> 11) + 1) * (1.0 / 9007199254740993.0);  // (0, 1]
        double u2 = (h2 >> 11) * (1.0 / 9007199254740992.0);        // [0, 1)
        double r = sqrt(-2.0 * log(u1));
        double s, c;
        sincospi(2.0 * u2, &s, &c);
        double d = 1.0 / (1.0 + kin[g]);
        X[band * npw + g] = make_double2(r * c * d, r * s * d);
    }
}

__global__ void damp_kernel(double2* X, long npw, const double* __restrict__ kin) {
    double2* x = X + (long)blockIdx.y * npw;
    for (long g = blockIdx.x * (long)blockDim.x + threadIdx.x; g < npw; g += (long)gridDim.x * blockDim.x) {
        double d = 1.0 / (1.0 + kin[g]);
        x[g] = make_double2(x[g].x * d, x[g].y * d);
    }
}

template <typename S2, typename T2>
__global__ void convert_kernel(const S2* __restrict__ in, T2* __restrict__ out, long count) {
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < count; t += (long)gridDim.x * blockDim.x)
        out[t] = conv<T2>(in[t]);
}

// a cluster of blocks per band: enough for two blocks on every SM, at least 1,024 values a block
template <typename... P, typename... A>
void launch_bands(fs_ctx* c, void (*kernel)(P...), int rows, A... args) {
    int cl = 1;
    while (cl < 8 && rows * cl < 2 * 152 && c->npw / (2 * cl) >= 1024) cl *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cl, rows);
    cfg.blockDim = dim3(RT);
    cfg.stream = c->stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    FS_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
}

inline int gx_for(long npw) { return (int)std::min<long>(64, (npw + 255) / 256); }

}  // namespace

template <typename T2>
void vec_resid(fs_ctx* c, const T2* X, const T2* Y, int m, double* resid, double2* dot, T2* RH) {
    if (m <= 0) return;
    ProfScope ps(c, ks_prec<T2>(KS_VECTOR), (RH ? 3.0 : 2.0) * m * c->npw * sizeof(T2), 16.0 * m * c->npw);
    launch_bands(c, resid_kernel<T2>, m, X, Y, (long)c->npw, resid, dot, RH);
}

template <typename T2>
void vec_resid_shift(fs_ctx* c, const T2* X, const T2* Y, const double* shift, int m, double* resid) {
    if (m <= 0) return;
    ProfScope ps(c, ks_prec<T2>(KS_VECTOR), 2.0 * m * c->npw * sizeof(T2), 8.0 * m * c->npw);
    launch_bands(c, resid_shift_kernel<T2>, m, X, Y, shift, (long)c->npw, resid);
}

template <typename T2>
void vec_make_w(fs_ctx* c, const T2* R, const int* act, int na, T2* W, double e_ref, double dE, int precond,
                const double* band_kin) {
    if (na <= 0) return;
    ProfScope ps(c, ks_prec<T2>(KS_VECTOR), 2.0 * na * c->npw * sizeof(T2) + c->npw * 8.0, 6.0 * na * c->npw);
    dim3 g(gx_for(c->npw), na);
    make_w_kernel<T2><<<g, 256, 0, c->stream>>>(R, act, c->npw, W, c->kin.as<double>(), e_ref, dE * dE, precond,
                                                 band_kin);
    FS_CUDA(cudaGetLastError());
}

template <typename T2>
void vec_a_resid(fs_ctx* c, const T2* ZR, T2* RH, const T2* X, const double2* dots, const double* theta, int m,
                 double* ra) {
    if (m <= 0) return;
    ProfScope ps(c, ks_prec<T2>(KS_VECTOR), 4.0 * m * c->npw * sizeof(T2), 20.0 * m * c->npw);
    launch_bands(c, a_resid_kernel<T2>, m, ZR, RH, X, dots, theta, (long)c->npw, ra);
}

// rows map[i] (or i) of X, and of Y when given, divided by the norm of X's row
template <typename T2> void vec_normalize(fs_ctx* c, T2* X, T2* Y, const int* map, int nrows) {
    if (nrows <= 0) return;
    ProfScope ps(c, ks_prec<T2>(KS_VECTOR), (Y ? 4.0 : 2.0) * nrows * c->npw * sizeof(T2), 6.0 * nrows * c->npw);
    launch_bands(c, normalize_kernel<T2>, nrows, X, Y, map, (long)c->npw);
}

template <typename T2> void vec_band_kin(fs_ctx* c, const T2* X, int m, double* out) {
    if (m <= 0) return;
    ProfScope ps(c, ks_prec<T2>(KS_VECTOR), 1.0 * m * c->npw * sizeof(T2) + 8.0 * c->npw, 6.0 * m * c->npw);
    band_kin_kernel<T2><<<m, RT, 0, c->stream>>>(X, c->kin.as<double>(), c->npw, out);
    FS_CUDA(cudaGetLastError());
}

void vec_damp_random(fs_ctx* c, double2* X, int m, int first, unsigned long long seed) {
    if (m - first <= 0) return;
    dim3 g(gx_for(c->npw), m - first);
    damp_random_kernel<<<g, 256, 0, c->stream>>>(X, c->npw, first, seed, c->kin.as<double>());
    FS_CUDA(cudaGetLastError());
}

void vec_damp(fs_ctx* c, double2* X, int m) {
    if (m <= 0) return;
    dim3 g(gx_for(c->npw), m);
    damp_kernel<<<g, 256, 0, c->stream>>>(X, c->npw, c->kin.as<double>());
    FS_CUDA(cudaGetLastError());
}

template <typename S2, typename T2> void vec_convert(fs_ctx* c, const S2* in, T2* out, size_t count) {
    if (count == 0) return;
    int b = (int)std::min<size_t>(4096, (count + 255) / 256);
    convert_kernel<S2, T2><<<b, 256, 0, c->stream>>>(in, out, (long)count);
    FS_CUDA(cudaGetLastError());
}

#define INST(T2)                                                                                           \
    template void vec_resid<T2>(fs_ctx*, const T2*, const T2*, int, double*, double2*, T2*);                \
    template void vec_resid_shift<T2>(fs_ctx*, const T2*, const T2*, const double*, int, double*);          \
    template void vec_make_w<T2>(fs_ctx*, const T2*, const int*, int, T2*, double, double, int, const double*); \
    template void vec_a_resid<T2>(fs_ctx*, const T2*, T2*, const T2*, const double2*, const double*, int,   \
                                  double*);                                                                 \
    template void vec_normalize<T2>(fs_ctx*, T2*, T2*, const int*, int);                                    \
    template void vec_band_kin<T2>(fs_ctx*, const T2*, int, double*);
INST(double2)
INST(float2)
template void vec_convert<double2, float2>(fs_ctx*, const double2*, float2*, size_t);
template void vec_convert<float2, double2>(fs_ctx*, const float2*, double2*, size_t);
