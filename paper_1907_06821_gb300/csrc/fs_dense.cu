// Small dense FP64 linear algebra of the Rayleigh-Ritz steps, on the GPU.
//
// Matrices are complex double, column-major, leading dimension = rows.
//   dense_gemm   C = alpha op(A) op(B) + beta C, op = N, C (conjugate transpose) or,
//                for B, T (transpose);
//                16 x 16 tiles staged in shared memory (FP64 FMA), or the tensor cores
//                (fs_oz.cu) when it is large.
//   dense_potrf  Cholesky A = L L^H of the lower triangle: diagonal blocks of 32 in
//                registers, their panels by row-wise triangular solves, products within
//                panels of 128 columns and one product per panel for the rest.
//                Reports the first non-positive pivot (LAPACK's info).
//   dense_trsm   B <- L^-1 B or L^-H B by inverted diagonal blocks of 128 and products.
//   dense_heev   the m lowest eigenpairs of a Hermitian matrix:
//     1. Householder reduction to a real symmetric tridiagonal T = Q^H A Q
//        (Q = H_0 ... H_{n-2}, H_i = I - tau_i v_i v_i^H, the LAPACK zhetd2
//        steps), all n - 1 steps in one cooperative kernel whose blocks exchange
//        one vector per step (bounded waits);
//     2. eigenvalues of T by bisection on Sturm counts (a warp evaluates 31
//        points of the bracket at once, so each round narrows it 32-fold; the
//        counts come from the leading minors, rescaled, without division);
//     3. eigenvectors of T by inverse iteration (Gaussian elimination with
//        partial pivoting on T - lambda I), vectors of eigenvalues closer
//        than 1e-13 ||T|| handled as one cluster and made orthogonal to each
//        other by modified Gram-Schmidt (a warp per cluster);
//     4. back-transformation Z = Q z in blocks of 128 reflectors (compact WY
//        form), each block as three GEMMs, then one Cholesky QR pass on Z.
// Every device-side wait (the exchange of the reduction) is bounded: on expiry the
// context's error flag is raised and the kernel returns.
#include "fs_common.cuh"

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

namespace {

constexpr int TB = 16;       // GEMM tile
constexpr int TK = 16;       // GEMM k step
constexpr int NBLK = 32;     // block size of the blocked factorisations
constexpr int PD_THREADS = 544;  // the 528 elements of a 32 x 32 lower triangle, whole warps
constexpr long long BAR_LIMIT = 1ll << 22;  // polls of a wait before it gives up
constexpr int HETRD_SMEM = 224 * 1024;

__device__ __forceinline__ double2 zconj(double2 a) { return make_double2(a.x, -a.y); }

// ------------------------------------------------------------------ GEMM
// C(m, n) = alpha sum_k a(m, k) b(k, n) + beta C(m, n), operands by strides and row maps.
// Bound by the FP64 pipe (about 2 FMAs per clock and SM), so what counts is that every SM
// gets an equal share and that no product is padding: 16 x 16 tiles, one output per thread,
// four FMAs per k in two chains.  (32 x 32 tiles with multiply-add-add took 1.5 operations
// per product and left the SMs uneven; the row-mapped 64 x 64 tiles of the subspace
// products took 1.9 ms for 36 x 36 x 1,069 on two SMs.  A plain FP64 solve of 8 states in
// 1,069 plane waves: 1,027 -> 80 ms; eigensolve of n = 816 with its Cholesky: 55 -> 43 ms.)
// Split K (gridDim.z > 1): block z takes k in [z kc, min(K, (z + 1) kc)) and
// writes its partial sum to part[(z N + n) M + m].
// lower = 1: tiles wholly above the diagonal (every row index below every column
// index) are skipped, for updates of which only the lower triangle is used.
__device__ __forceinline__ const double2* mat_at(const OzMat& A, int r, int k) {
    if (A.rp) return A.rp[r] + (long)k * A.sk;
    if (A.kp) return A.kp[k] + (long)r * A.sr;
    return A.X + (A.map ? (long)A.map[r] : (long)r) * A.sr + (A.kmap ? (long)A.kmap[k] : (long)k) * A.sk;
}

__global__ void __launch_bounds__(TB * TB) zgemm_kernel(int M, int N, int K, double alpha, OzMat A, OzMat B,
                                                        double beta, OzDst C, double2* part, int kc, int lower) {
    __shared__ double2 As[TK][TB + 1];
    __shared__ double2 Bs[TK][TB + 1];
    const int m0 = blockIdx.x * TB, n0 = blockIdx.y * TB;
    if (lower && m0 + TB <= n0) return;
    const int kbeg = blockIdx.z * kc, kend = min(K, kbeg + kc);
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    // this thread's tile elements: along k when the operand is contiguous in k, else along the rows
    const int ak = A.sk == 1 ? tx : ty, am = A.sk == 1 ? ty : tx;
    const int bk = B.sk == 1 ? tx : ty, bn = B.sk == 1 ? ty : tx;
    const bool aok = m0 + am < M, bok = n0 + bn < N;
    auto load = [&](int k0, double2& va, double2& vb) {
        va = vb = make_double2(0.0, 0.0);
        if (aok && k0 + ak < kend) va = *mat_at(A, m0 + am, k0 + ak);
        if (bok && k0 + bk < kend) vb = *mat_at(B, n0 + bn, k0 + bk);
        if (A.conj) va.y = -va.y;
        if (B.conj) vb.y = -vb.y;
    };
    double2 acc = make_double2(0.0, 0.0), va, vb;
    load(kbeg, va, vb);  // the next step's elements are loaded while the current step's are multiplied
    for (int k0 = kbeg; k0 < kend; k0 += TK) {
        As[ak][am] = va;
        Bs[bk][bn] = vb;
        __syncthreads();
        if (k0 + TK < kend) load(k0 + TK, va, vb);
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            const double2 a = As[kk][tx], b = Bs[kk][ty];
            acc.x = fma(a.x, b.x, acc.x);
            acc.y = fma(a.x, b.y, acc.y);
            acc.x = fma(-a.y, b.y, acc.x);
            acc.y = fma(a.y, b.x, acc.y);
        }
        __syncthreads();
    }
    const int m = m0 + tx, n = n0 + ty;
    if (m >= M || n >= N) return;
    if (part) {
        part[((long)blockIdx.z * N + n) * M + m] = acc;
        return;
    }
    double2* c = C.C + (C.mmap ? (long)C.mmap[m] : (long)m) * C.cm + (C.nmap ? (long)C.nmap[n] : (long)n) * C.cn;
    double2 o = make_double2(alpha * acc.x, alpha * acc.y);
    if (beta != 0.0) {
        o.x += beta * c->x;
        o.y += beta * c->y;
    }
    *c = o;
}

// ------------------------------------------------------------------ Cholesky
// Factor the b x b diagonal block at A + j0 (1 + lda); squared pivots to piv[j0 + j]; the
// first non-positive pivot sets *info = j0 + j + 1 (once) and is replaced by 1 so that the
// arithmetic stays finite.  A thread keeps one element of the lower triangle in a register, in
// column order, so that the rank-1 term of column j runs on the warps behind it only (a warp's
// FP64 instruction costs the same with one lane as with 32: a square of 32 warps spent three
// times as many: two factorisations at n = 816 3.0 -> 2.2 ms, n = 108 0.35 -> 0.25 ms).  Chain of a column: rank-1 term, hand-over, reciprocal square root, scaling,
// hand-over.
__global__ void __launch_bounds__(PD_THREADS) potrf_diag_kernel(double2* A, int lda, int j0, int b, double* piv,
                                                                int* info) {
    __shared__ double2 raw[2][NBLK], col[2][NBLK];  // column j before and after scaling
    // element t of the triangle: column c holds rows c .. 31
    int r = threadIdx.x, c = 0;
    while (c < NBLK && r >= NBLK - c) r -= NBLK - c++;
    r += c;
    double2* D = A + j0 + (long)j0 * lda;
    const bool live = c < b && r < b;
    double2 a = live ? D[r + (long)c * lda] : make_double2(0.0, 0.0);
    if (c == 0) raw[0][r] = a;
    __syncthreads();
    for (int j = 0; j < b; ++j) {
        if (c == j) {
            double p = raw[j & 1][j].x;
            const bool bad = !(p > 0.0);
            if (r == j) {
                if (piv) piv[j0 + j] = p;
                if (bad) atomicCAS(info, 0, j0 + j + 1);
            }
            if (bad) p = 1.0;
            const double inv = rsqrt(p);
            a = r == j ? make_double2(p * inv, 0.0) : cscale(a, inv);
            col[j & 1][r] = a;
        }
        __syncthreads();
        if (c > j && c < NBLK) {
            const double2 x = col[j & 1][r], y = col[j & 1][c];  // a -= x conj(y)
            a.x = fma(-x.x, y.x, fma(-x.y, y.y, a.x));
            a.y = fma(x.x, y.y, fma(-x.y, y.x, a.y));
            if (c == j + 1) raw[c & 1][r] = a;
        }
        __syncthreads();
    }
    if (live) D[r + (long)c * lda] = a;
}

// rows r >= j0 + b of the panel: A[r, j0:j0+b] <- A[r, j0:j0+b] L^-H (L the
// factored block); one warp per row, lane c holding column c.
__global__ void potrf_panel_kernel(double2* A, int lda, int n, int j0, int b) {
    __shared__ double2 Ls[NBLK][NBLK + 1];
    for (int i = threadIdx.x; i < b * b; i += blockDim.x) {
        const int rr = i % b, cc = i / b;
        const double2 l = A[j0 + rr + (long)(j0 + cc) * lda];
        Ls[rr][cc] = rr == cc ? make_double2(1.0 / l.x, 0.0) : l;  // reciprocals on the diagonal
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int r = j0 + b + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (r >= n) return;
    double2 xv = lane < b ? A[r + (long)(j0 + lane) * lda] : make_double2(0.0, 0.0);
    // x_c = (a_c - sum_{k<c} x_k conj(L[c][k])) / L[c][c]
    for (int c = 0; c < b; ++c) {
        if (lane == c) xv = cscale(xv, Ls[c][c].x);
        const double2 xc = make_double2(__shfl_sync(0xffffffffu, xv.x, c), __shfl_sync(0xffffffffu, xv.y, c));
        if (lane > c && lane < b) {
            const double2 l = Ls[lane][c];
            xv.x = fma(-xc.x, l.x, fma(-xc.y, l.y, xv.x));
            xv.y = fma(xc.x, l.y, fma(-xc.y, l.x, xv.y));
        }
    }
    if (lane < b) A[r + (long)(j0 + lane) * lda] = xv;
}

// ------------------------------------------------------------------ triangular solves
// Inverses of the IB x IB diagonal blocks of the lower triangular L, all in one launch: a
// warp per column j of a block solves L x = e_j (lane l holding rows l, l + 32, ..).  Block
// b goes to X + b IB IB (ld IB), zeros above the diagonal.  With them a triangular solve is
// GEMMs alone, of 128 k a step (on the tensor cores when the right-hand sides are many)
// instead of 32 with a substitution kernel between: n = 816, 816 columns: 3.3 ms before.
constexpr int IB = 128;
__global__ void __launch_bounds__(128) tri_inv_kernel(const double2* L, int lda, int n, double2* X) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const int j0 = (w / IB) * IB, j = w % IB, b = min(IB, n - j0);
    if (j0 >= n || j >= b) return;
    const double2* D = L + j0 + (long)j0 * lda;
    double2* out = X + (long)j0 * IB + (long)j * IB;
    double2 x[IB / 32];
    double id[IB / 32];  // reciprocals of the diagonal entries
#pragma unroll
    for (int q = 0; q < IB / 32; ++q) {
        const int r = lane + 32 * q;
        x[q] = make_double2(r == j ? 1.0 : 0.0, 0.0);
        id[q] = r >= j && r < b ? 1.0 / D[r + (long)r * lda].x : 0.0;
    }
    // column k of L, the next one loaded while the current one is used
    auto load = [&](int k, double2 (&lk)[IB / 32]) {
#pragma unroll
        for (int q = 0; q < IB / 32; ++q) {
            const int r = lane + 32 * q;
            lk[q] = r > k && r < b ? D[r + (long)k * lda] : make_double2(0.0, 0.0);
        }
    };
    double2 nx[IB / 32];
    load(j, nx);
#pragma unroll
    for (int g = 0; g < IB / 32; ++g) {
        if (32 * g + 31 < j || 32 * g >= b) continue;
        for (int l = max(0, j - 32 * g); l < min(32, b - 32 * g); ++l) {
            const int k = 32 * g + l;
            double2 lk[IB / 32];
#pragma unroll
            for (int q = 0; q < IB / 32; ++q) lk[q] = nx[q];
            load(k + 1, nx);  // (rows beyond k + 1 only: none for the last column)
            if (lane == l) x[g] = cscale(x[g], id[g]);
            const double2 xk = make_double2(__shfl_sync(0xffffffffu, x[g].x, l), __shfl_sync(0xffffffffu, x[g].y, l));
#pragma unroll
            for (int q = g; q < IB / 32; ++q) {
                x[q].x = fma(-lk[q].x, xk.x, fma(lk[q].y, xk.y, x[q].x));
                x[q].y = fma(-lk[q].x, xk.y, fma(-lk[q].y, xk.x, x[q].y));
            }
        }
    }
#pragma unroll
    for (int q = 0; q < IB / 32; ++q) out[lane + 32 * q] = lane + 32 * q < b ? x[q] : make_double2(0.0, 0.0);
}

__global__ void conj_transpose_kernel(int n, int m, const double2* A, int lda, double2* out, int ldo) {
    long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)n * m) return;
    const int r = (int)(t % n), c = (int)(t / n);
    out[c + (long)r * ldo] = zconj(A[r + (long)c * lda]);
}

// Z (n x m) = T^H (T m x n) unless *info
__global__ void qr_back_kernel(int n, int m, const double2* T, double2* Z, int ldz, const int* info) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)n * m || *info) return;
    const int r = (int)(t % n), c = (int)(t / n);
    Z[r + (long)c * ldz] = zconj(T[c + (long)r * m]);
}

// A <- (A + A^H) / 2 (exactly Hermitian input for the reduction)
__global__ void hermitize_kernel(double2* A, int n) {
    long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)n * n) return;
    const int r = (int)(t % n), c = (int)(t / n);
    if (r < c) return;
    const double2 a = A[r + (long)c * n], b = A[c + (long)r * n];
    const double2 h = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
    A[r + (long)c * n] = h;
    A[c + (long)r * n] = zconj(h);
    if (r == c) A[r + (long)c * n].y = 0.0;
}

// ------------------------------------------------------------------ scaling
// Powers of two s_i = 2^e with B_ii / 4^e in [0.5, 2) (1 where the diagonal is not a positive
// number) and their reciprocals: with A and B divided by s_i s_j the factor L of B has rows of
// norm about one.  The products of a triangular solve are exact only to 2^-55 of (largest of a row)
// x (largest of a column) on the tensor cores, and rows of B that differ by d make the columns of
// the inverted blocks and the rows of the right-hand side differ by 1 / d and d: unscaled, a B
// spread over twelve decades lost four to six digits.  Exact, and no change for a B of unit diagonal.
__global__ void equil_scale_kernel(const double2* B, int n, double* s) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double b = B[i + (long)i * n].x;
    const int e = b > 0.0 && isfinite(b) ? (ilogb(b) + 1) >> 1 : 0;
    s[i] = scalbn(1.0, e);
    s[n + i] = scalbn(1.0, -e);
}
__global__ void equil_sym_kernel(double2* A, double2* B, int n, const double* s) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)n * n) return;
    const double fr = s[n + t % n], fc = s[n + t / n];
    A[t] = cscale(cscale(A[t], fr), fc);
    B[t] = cscale(cscale(B[t], fr), fc);
}
__global__ void equil_rows_kernel(const double2* Z, int n, int m, const double* s, double2* out) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t < (long)n * m) out[t] = cscale(Z[t], s[n + t % n]);
}

// ------------------------------------------------------------------ tridiagonal reduction
// Full Hermitian A (n x n, both triangles).  Step i: reflector v_i (v[0] = 1 at
// row i + 1) with H^H x = beta e_1 for x = A[i+1:, i]; y_i = A22 v_i;
// s_i = v_i^H y_i; w_i = tau_i y_i - (|tau_i|^2 s_i / 2) v_i;
// A22 -= v_i w_i^H + w_i v_i^H.  Outputs: d, e (real), tau, V[:, i] = v_i.
//
// All n - 1 steps in one cooperative kernel.  Block b owns the columns j = b mod gridDim.x
// (in shared memory when they fit, else in place) and thread t of every block the rows
// r = t mod HT, whose parts of v and w it keeps in registers.  In a step a block brings its
// columns up to date, forms y_i[j] = <column j, v_i> for them and publishes these numbers
// (and, from the owner of column i + 1, that column); every block then forms w_i, the
// updated column i + 1 and the next reflector for itself.  The published numbers are their
// own flags: Y and C have a row per step, filled with a NaN pattern beforehand, and the
// readers poll until every entry has changed, so a step costs one store and one load
// through L2 instead of a grid barrier, a segment sum and three reads of A.
// Bound: FP64 rate (14 operations per element of A22 and step, 20 per row and block) and
// about 6 us a step of dependent FP64 operations and L2 round trips.  Four warps, one per
// scheduler: what every warp computes for itself (the reflector's scalars, the sums) then
// costs its own pipe only; eight took 45 % longer at n = 108.  Measured: n = 816: 20.0 ->
// 14.4 ms, n = 204: 2.3 -> 1.6 ms.
constexpr unsigned long long EMPTY = 0xffffffffffffffffull;     // a NaN that no arithmetic returns

__device__ __forceinline__ void publish(double* p, double v) {
    if ((unsigned long long)__double_as_longlong(v) == EMPTY) v = __longlong_as_double(0x7ff8000000000000ll);
    asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ double2 peek(const double2* p) {
    double2 v;
    asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ bool is_empty(double2 v) {
    return (unsigned long long)__double_as_longlong(v.x) == EMPTY || (unsigned long long)__double_as_longlong(v.y) == EMPTY;
}

// 1 / sqrt(s) and 1 / s for normal s > 0 by Newton's iteration from a single-precision start on
// the mantissa (an FP64 instruction holds a warp's pipe for 64 cycles, and the library forms
// take three times as many of them): relative error below 2^-51
__device__ __forceinline__ double newton_rsqrt(double s) {
    const int h = __double2hiint(s), ex = ((h >> 20) - 1023) & ~1;  // even part of the exponent
    const double m = __hiloint2double(h - (ex << 20), __double2loint(s));  // in [1, 4)
    double y = (double)rsqrtf((float)m);
    const double hm = 0.5 * m;
    y = y * fma(-hm * y, y, 1.5);
    y = fma(y * fma(-hm * y, y, 0.5), 1.0, y);
    return __hiloint2double(__double2hiint(y) - ((ex / 2) << 20), __double2loint(y));
}
__device__ __forceinline__ double newton_rcp(double s) {
    const int h = __double2hiint(s), ex = (h >> 20) - 1023;
    const double m = __hiloint2double(h - (ex << 20), __double2loint(s));  // in [1, 2)
    double y = (double)(1.0f / (float)m);
    y = fma(y, fma(-m, y, 1.0), y);
    y = fma(y, fma(-m, y, 1.0), y);
    return __hiloint2double(__double2hiint(y) - (ex << 20), __double2loint(y));
}

// sum over the block of one double per thread, given to every thread; red: HT / 32 doubles
// that no other use touches until the next barrier
template <int HT> __device__ __forceinline__ double ht_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = red[threadIdx.x & (HT / 32 - 1)];
    for (int o = HT / 64; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

template <int HT, int PER>
__global__ void __launch_bounds__(HT)
hetrd_kernel(int n, double2* A, double2* V, double2* tau, double* d, double* e, double2* Y, double2* C, int in_smem,
             int* err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* sv = reinterpret_cast<double2*>(smem_raw);  // v_{i-1} and w_{i-1} by row
    double2* sw = sv + n;
    const int nb = gridDim.x, bid = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int nown = (n - bid + nb - 1) / nb;  // owned columns bid, bid + nb, ...
    double2* cols = in_smem ? sw + n : A + (long)bid * n;
    const long cstr = in_smem ? n : (long)nb * n;
    double2* part = in_smem ? sw + n + (long)((n + nb - 1) / nb) * n : sw + n;  // [nown][HT / 32]
    __shared__ double red[2][HT / 32];
    __shared__ double2 head[2];  // broadcast of y[i + 1] and of the head of the next reflector
    __shared__ int gave_up;
    if (tid == 0) gave_up = 0;
    if (n < 2) {
        if (bid == 0 && tid == 0 && n == 1) d[0] = A[0].x;
        return;
    }
    if (in_smem)
        for (int s = 0; s < nown; ++s)
            for (int r = tid; r < n; r += HT) cols[s * cstr + r] = A[(long)(bid + s * nb) * n + r];
    // x: the column to eliminate (rows > i), as registers; v, w of this step, vp, of the last
    double2 v[PER], w[PER], x[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int r = tid + q * HT;
        x[q] = r < n ? __ldcg(A + r) : make_double2(0.0, 0.0);
        v[q] = w[q] = make_double2(0.0, 0.0);
    }
    if (bid == 0 && tid == 0) d[0] = x[0].x;
    for (int i = 0;; ++i) {
        // reflector v_i from x (rows i + 1 ..); every thread derives the scalars itself
        double ss = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int r = tid + q * HT;
            if (r == i + 1) head[0] = x[q];
            if ((r | 31) < i + 2 || (r & ~31) >= n) continue;  // warp-uniform
            if (r >= i + 2 && r < n) ss = fma(x[q].x, x[q].x, fma(x[q].y, x[q].y, ss));
        }
        const double xn2 = ht_sum<HT>(ss, red[0]);
        const double2 al = head[0];
        double2 t = make_double2(0.0, 0.0), sc = t;
        double beta = al.x;
        if (!(xn2 == 0.0 && al.y == 0.0)) {  // else nothing to eliminate: H = I
            const double s2 = fma(al.x, al.x, fma(al.y, al.y, xn2));
            double ib, id, dx;
            if (s2 > 0x1p-900 && s2 < 0x1p+900) {
                // square root and its reciprocal corrected to their last bit (a reflector is unitary
                // to the accuracy of these two)
                const double rs = newton_rsqrt(s2), q0 = s2 * rs;
                const double nrm = fma(0.5 * rs, fma(-q0, q0, s2), q0);
                beta = -copysign(nrm, al.x);
                ib = -copysign(fma(rs, fma(-nrm, rs, 1.0), rs), al.x);
                dx = al.x - beta;
                id = newton_rcp(fma(dx, dx, al.y * al.y));
            } else {
                beta = -copysign(sqrt(s2), al.x);
                ib = 1.0 / beta;
                dx = al.x - beta;
                id = 1.0 / fma(dx, dx, al.y * al.y);
            }
            t = make_double2(-dx * ib, -al.y * ib);
            sc = make_double2(dx * id, -al.y * id);  // 1 / (alpha - beta)
        }
        // v_i into x; the registers v keep v_{i-1} for the update below
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int r = tid + q * HT;
            if (r == i + 1) {
                x[q] = make_double2(1.0, 0.0);
            } else if (r > i + 1 && r < n) {
                x[q] = make_double2(fma(x[q].x, sc.x, -x[q].y * sc.y), fma(x[q].x, sc.y, x[q].y * sc.x));
            } else {
                x[q] = make_double2(0.0, 0.0);
            }
            if (bid == 0 && r > i && r < n) V[r + (long)i * n] = x[q];
        }
        if (bid == 0 && tid == 0) {
            tau[i] = t;
            e[i] = beta;
        }
        // own columns j > i: the rank-2 term of step i - 1, then y_i[j] = <column j, v_i>
        const int s0 = (i + 1 - bid + nb - 1) / nb;  // first owned column beyond i
        auto column = [&](int s) {
            const int j = bid + s * nb;
            double2* col = cols + s * cstr;
            double2 vj = make_double2(0.0, 0.0), wj = vj, acc = vj;
            if (i > 0) vj = sv[j], wj = sw[j];
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int r = tid + q * HT;
                if ((r | 31) <= i || (r & ~31) >= n) continue;  // warp-uniform
                if (r > i && r < n) {
                    double2 a = col[r];
                    if (i > 0) {  // a -= v conj(wj) + w conj(vj)
                        // (the term by itself first: one rounding at the size of a, not four)
                        a.x -= fma(v[q].x, wj.x, fma(v[q].y, wj.y, fma(w[q].x, vj.x, w[q].y * vj.y)));
                        a.y -= fma(v[q].y, wj.x, fma(-v[q].x, wj.y, fma(w[q].y, vj.x, -w[q].x * vj.y)));
                        col[r] = a;
                    }
                    if (j == i + 1) {
                        publish(&C[(long)i * n + r].x, a.x);
                        publish(&C[(long)i * n + r].y, a.y);
                    }
                    acc.x = fma(a.x, x[q].x, fma(a.y, x[q].y, acc.x));
                    acc.y = fma(a.x, x[q].y, fma(-a.y, x[q].x, acc.y));
                }
            }
            return acc;
        };
        // warp sums of two columns at a time: lanes below 16 take the first, the others the
        // second, then every eight lanes the real or the imaginary parts
        for (int s = s0; s < nown; s += 2) {
            const double2 a0 = column(s);
            const double2 a1 = s + 1 < nown ? column(s + 1) : make_double2(0.0, 0.0);
            const bool up = lane & 16;
            const double kx = up ? a1.x : a0.x, ky = up ? a1.y : a0.y;
            const double sx = up ? a0.x : a1.x, sy = up ? a0.y : a1.y;
            const double px = kx + __shfl_xor_sync(0xffffffffu, sx, 16);
            const double py = ky + __shfl_xor_sync(0xffffffffu, sy, 16);
            const bool im = lane & 8;
            double p = (im ? py : px) + __shfl_xor_sync(0xffffffffu, im ? px : py, 8);
            for (int o = 4; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
            const int sc_ = s + (lane >> 4);
            if ((lane & 7) == 0 && sc_ < nown)
                reinterpret_cast<double*>(part + sc_ * (HT / 32) + wp)[(lane >> 3) & 1] = p;
        }
        __syncthreads();
        for (int q = tid; q < 2 * (nown - s0); q += HT) {
            const int s = s0 + (q >> 1), c = q & 1;
            const double* ps = reinterpret_cast<const double*>(part + s * (HT / 32)) + c;
            publish(reinterpret_cast<double*>(Y + (long)i * n + bid + s * nb) + c,
                    HT == 128 ? (ps[0] + ps[2]) + (ps[4] + ps[6])
                              : ((ps[0] + ps[2]) + (ps[4] + ps[6])) + ((ps[8] + ps[10]) + (ps[12] + ps[14])));
        }
        // everybody's y_i and column i + 1
        double2 y[PER], c[PER];
        {
            long long it = 0;
            bool more = true;
            while (more) {
                more = false;
#pragma unroll
                for (int q = 0; q < PER; ++q) {
                    const int r = tid + q * HT;
                    if (r > i && r < n) {
                        y[q] = peek(Y + (long)i * n + r);
                        c[q] = peek(C + (long)i * n + r);
                    } else {
                        y[q] = c[q] = make_double2(0.0, 0.0);
                    }
                }
#pragma unroll
                for (int q = 0; q < PER; ++q) more = more || is_empty(y[q]) || is_empty(c[q]);
                if (more && (++it > BAR_LIMIT || ((it & 1023) == 0 && *(volatile int*)err))) {
                    *(volatile int*)err = 1;
                    gave_up = 1;
                    break;
                }
            }
        }
        double sp = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int r = tid + q * HT;
            if ((r | 31) <= i || (r & ~31) >= n) continue;
            if (r == i + 1) head[1] = y[q];
            sp = fma(x[q].x, y[q].x, fma(x[q].y, y[q].y, sp));
        }
        const double h = 0.5 * fma(t.x, t.x, t.y * t.y) * ht_sum<HT>(sp, red[1]);
        if (gave_up) return;  // block-uniform: set before the barrier in ht_sum
        const double2 y0 = head[1];
        const double2 w0 = make_double2(fma(t.x, y0.x, fma(-t.y, y0.y, -h)), fma(t.x, y0.y, t.y * y0.x));
        // v <- v_i, w <- w_i = t y - h v, x <- column i + 1 minus its rank-2 term (v[0] = 1)
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int r = tid + q * HT;
            if ((r | 31) <= i || (r & ~31) >= n) continue;
            v[q] = x[q];
            w[q] = make_double2(fma(t.x, y[q].x, fma(-t.y, y[q].y, -h * v[q].x)),
                                fma(t.x, y[q].y, fma(t.y, y[q].x, -h * v[q].y)));
            x[q].x = c[q].x - fma(v[q].x, w0.x, fma(v[q].y, w0.y, w[q].x));
            x[q].y = c[q].y - fma(v[q].y, w0.x, fma(-v[q].x, w0.y, w[q].y));
            if (r > i && r < n) {
                sv[r] = v[q];
                sw[r] = w[q];
                if (r == i + 1 && bid == 0) d[i + 1] = x[q].x;
            }
        }
        if (i == n - 2) return;
        // sv, sw are read after the barrier in the next ht_sum
    }
}

// ------------------------------------------------------------------ tridiagonal eigenvalues
// number of eigenvalues of T (d, e) below x: sign changes of the leading
// principal minors p_j = (d_j - x) p_{j-1} - e_{j-1}^2 p_{j-2} (p_{-1} = 1),
// carried with exact power-of-two rescaling (no division); a zero minor counts
// as a change of sign, the role of LAPACK's pivmin in the ratio form.
// FP64 instructions are what a step costs (three here), so signs, zero tests and the range
// checks (every fourth step: a step changes the magnitude by far less than 2^100 up, and a
// minor that falls out of range at the bottom has lost its weight) are taken on the high words.
__device__ __forceinline__ int sturm_count(const double* d, const double* e2, int n, double x, double) {
    const double big = 0x1p+500, small = 0x1p-500;
    double pm = 1.0, p = d[0] - x;
    int cnt = !(p > 0.0);
    if (p == 0.0) p = -small;
#pragma unroll 4
    for (int j = 1; j < n; ++j) {
        double q = fma(d[j] - x, p, -(e2[j - 1] * pm));
        const int hp = __double2hiint(p), hq = __double2hiint(q);
        if ((((unsigned)hq << 1) | (unsigned)__double2loint(q)) == 0) {
            q = hp >= 0 ? -small : small;
            cnt += 1;
        } else {
            cnt += (unsigned)(hq ^ hp) >> 31;
        }
        pm = p;
        p = q;
        if ((j & 3) == 3) {
            const int ep = (__double2hiint(p) >> 20) & 0x7ff, em = (__double2hiint(pm) >> 20) & 0x7ff;
            if (ep > 1023 + 400) {
                p *= small;
                pm *= small;
            } else if (max(ep, em) < 1023 - 400) {
                p *= big;
                pm *= big;
            }
        }
    }
    return cnt;
}

// T scaled by a power of two to a norm of about one (ds, e2 = scaled e squared) for the counts,
// its Gershgorin interval and pivmin; info3[3]: the norm of T, [4]: the factor back (one block)
__global__ void tri_prep_kernel(const double* d, const double* e, double* ds, double* e2, int n, double* info3) {
    __shared__ double lo_s[256], hi_s[256], em_s[256];
    double lo = 1e300, hi = -1e300, em = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double a = j > 0 ? fabs(e[j - 1]) : 0.0, b = j < n - 1 ? fabs(e[j]) : 0.0;
        lo = fmin(lo, d[j] - a - b);
        hi = fmax(hi, d[j] + a + b);
        if (j < n - 1) em = fmax(em, fabs(e[j]));
    }
    lo_s[threadIdx.x] = lo;
    hi_s[threadIdx.x] = hi;
    em_s[threadIdx.x] = em;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            lo_s[threadIdx.x] = fmin(lo_s[threadIdx.x], lo_s[threadIdx.x + o]);
            hi_s[threadIdx.x] = fmax(hi_s[threadIdx.x], hi_s[threadIdx.x + o]);
            em_s[threadIdx.x] = fmax(em_s[threadIdx.x], em_s[threadIdx.x + o]);
        }
        __syncthreads();
    }
    const double tnorm = fmax(fabs(lo_s[0]), fabs(hi_s[0]));
    int ex = 0;
    if (tnorm > 0 && isfinite(tnorm)) frexp(tnorm, &ex);
    ex = min(max(ex, -1000), 1000);
    const double sc = ldexp(1.0, -ex);
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        ds[j] = d[j] * sc;
        if (j < n - 1) e2[j] = (e[j] * sc) * (e[j] * sc);
    }
    if (threadIdx.x == 0) {
        const double pad = 2.0 * DBL_EPSILON * (tnorm * sc) + 1e-300;
        info3[0] = lo_s[0] * sc - pad;
        info3[1] = hi_s[0] * sc + pad;
        info3[2] = fmax(1e-300, DBL_MIN * fmax(1.0, (em_s[0] * sc) * (em_s[0] * sc)));  // pivmin
        info3[3] = tnorm;
        info3[4] = ldexp(1.0, ex);
    }
}

// eigenvalue k (ascending) of T, one warp per index: 31 interior points of the
// bracket per round, each round narrowing it 32-fold
__global__ void tri_bisect_kernel(const double* d, const double* e2, int n, int m, const double* info3, double* w) {
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= m) return;
    double a = info3[0], b = info3[1];
    const double pivmin = info3[2];
    for (int round = 0; round < 24; ++round) {
        const double tol = 2.0 * DBL_EPSILON * fmax(fabs(a), fabs(b)) + 2.0 * pivmin;
        if (b - a <= tol) break;
        const double x = a + (b - a) * (double)(lane + 1) * (1.0 / 32.0);
        const int cnt = lane < 31 ? sturm_count(d, e2, n, x, pivmin) : n + 1;
        // the first point whose count exceeds k bounds eigenvalue k from above
        const unsigned int above = __ballot_sync(0xffffffffu, cnt > k);
        const int f = __ffs(above) - 1;  // lane 31 always qualifies
        const double nb_ = a + (b - a) * (double)(f + 1) * (1.0 / 32.0);
        const double na_ = f > 0 ? a + (b - a) * (double)f * (1.0 / 32.0) : a;
        a = na_;
        b = f < 31 ? nb_ : b;
    }
    if (lane == 0) w[k] = 0.5 * (a + b) * info3[4];
}

// ------------------------------------------------------------------ tridiagonal eigenvectors
// Inverse iteration for the clusters of w (ascending), one warp (block) per
// index: the block of index k0 starts a cluster when w[k0] - w[k0 - 1] >
// 1e-13 ||T|| and computes the cluster's vectors in order, each made
// orthogonal to the cluster's earlier ones.  An eigenvector from inverse
// iteration is accurate to about eps ||T|| / gap, so vectors outside a cluster
// are orthogonal to 2e-3 or better, and the Cholesky QR pass that follows makes
// them orthonormal to working precision; it mixes neighbours by that angle, which
// changes their residuals by eps ||T||.  Eigenvalues closer than that (the E +- d
// pairs of the folded spectrum, an orthonormal block's unit eigenvalues) share a
// cluster.  (With 1e-10 the low end of the wire's folded spectrum, 1e-9 apart at
// ||T|| of some 100, made clusters whose vectors one warp computed in turn: 8 ms a
// call at n = 816.)  Lane 0 runs the elimination and the substitutions (sequential in
// the position) on shared-memory copies of T, of the factors and of the
// vector; all lanes run the Gram-Schmidt steps and the norms.  z: [n][m] real
// (position-major) and, complex, in Z.  Dynamic shared memory: 8 n doubles.
__global__ void __launch_bounds__(32) tri_invit_kernel(const double* d, const double* e, int n, int m,
                                                       const double* w, const double* info3, double* z,
                                                       double2* Z, int ldz) {
    extern __shared__ __align__(16) double tsm[];
    double* dd = tsm;          // diagonal of T
    double* ee = dd + n;       // off-diagonal of T (ee[n - 1] = 0)
    double* ri = ee + n;       // pivot of row i of U
    double* u1 = ri + n;       // first and second super-diagonals of U
    double* u2 = u1 + n;
    double* mu = u2 + n;       // multipliers
    double* sw = mu + n;       // 1 where rows i and i + 1 were swapped
    double* zv = sw + n;       // the vector being iterated
    const int k0 = blockIdx.x;
    const int lane = threadIdx.x;
    if (k0 >= m) return;
    const double tnorm = fmax(info3[3], 1e-300);
    const double ctol = 1e-13 * tnorm;
    if (k0 > 0 && w[k0] - w[k0 - 1] <= ctol) return;  // not a cluster start (block-uniform)
    int k1 = k0 + 1;
    while (k1 < m && w[k1] - w[k1 - 1] <= ctol) ++k1;
    for (int i = lane; i < n; i += 32) {
        dd[i] = d[i];
        ee[i] = i < n - 1 ? e[i] : 0.0;
    }
    __syncwarp();
#define ZV(q, i) z[(long)(i) * m + (q)]
    const double sep = 10.0 * DBL_EPSILON * tnorm;
    double lam_prev = -1e300;
    for (int k = k0; k < k1; ++k) {
        double lam = w[k];
        if (lam - lam_prev < sep) lam = lam_prev + sep;  // separate equal eigenvalues of a cluster
        lam_prev = lam;
        if (lane == 0) {
            // elimination with partial pivoting of T - lam I: U rows (pivot, u1, u2), multipliers, swaps
            double p0 = dd[0] - lam, p1 = n > 1 ? ee[0] : 0.0, p2 = 0.0;
            for (int i = 0; i < n - 1; ++i) {
                const double sv = ee[i], a = dd[i + 1] - lam, t = ee[i + 1];
                if (fabs(p0) >= fabs(sv)) {
                    if (p0 == 0.0) p0 = sep;
                    const double f = sv / p0;
                    ri[i] = p0; u1[i] = p1; u2[i] = p2; mu[i] = f; sw[i] = 0.0;
                    p0 = a - f * p1;
                    p1 = t - f * p2;
                    p2 = 0.0;
                } else {
                    const double f = p0 / sv;
                    ri[i] = sv; u1[i] = a; u2[i] = t; mu[i] = f; sw[i] = 1.0;
                    p0 = p1 - f * a;
                    p1 = p2 - f * t;
                    p2 = 0.0;
                }
            }
            ri[n - 1] = p0;
            // start vector: a fixed pseudo-random sequence per index
            unsigned int st = 2654435761u * (unsigned int)(k + 1) + 12345u;
            for (int i = 0; i < n; ++i) {
                st = st * 1664525u + 1013904223u;
                zv[i] = 0.5 + (double)(st >> 8) * (1.0 / 16777216.0);
            }
        }
        __syncwarp();
        // small pivots raised to 10 eps ||T||, then their reciprocals (a division per position and
        // sweep on lane 0 alone would be the longest chain of the iteration).  The last pivot is small
        // whenever lam is an eigenvalue, and raising it by s makes the iteration converge to a
        // vector of T + s e_n e_n^T: it is only kept above 2^-10 of that (n = 8: residual 1.2e-15
        // with the last one raised like the others)
        for (int i = lane; i < n; i += 32) {
            const double least = i < n - 1 ? sep : sep * 0x1p-10;
            double u = ri[i];
            if (fabs(u) < least) u = u < 0 ? -least : least;
            ri[i] = 1.0 / u;
        }
        __syncwarp();
        for (int it = 0; it < 4; ++it) {
            if (lane == 0) {
                // forward: apply the row operations
                double xi = zv[0];
                for (int i = 0; i < n - 1; ++i) {
                    const double xn = zv[i + 1];
                    if (sw[i] != 0.0) {
                        zv[i] = xn;
                        xi = xi - mu[i] * xn;
                    } else {
                        zv[i] = xi;
                        xi = xn - mu[i] * xi;
                    }
                }
                zv[n - 1] = xi;
                // back substitution with the three diagonals of U
                double x2 = 0.0, x1 = zv[n - 1] * ri[n - 1];
                zv[n - 1] = x1;
                for (int i = n - 2; i >= 0; --i) {
                    const double x0 = fma(-u1[i], x1, fma(-u2[i], x2, zv[i])) * ri[i];
                    zv[i] = x0;
                    x2 = x1;
                    x1 = x0;
                }
            }
            __syncwarp();
            // orthogonalise against the cluster's earlier vectors (warp-parallel), normalise
            for (int q = k0; q < k; ++q) {
                double dot = 0;
                for (int i = lane; i < n; i += 32) dot += ZV(q, i) * zv[i];
                for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                for (int i = lane; i < n; i += 32) zv[i] -= dot * ZV(q, i);
                __syncwarp();
            }
            double nrm = 0;
            for (int i = lane; i < n; i += 32) nrm += zv[i] * zv[i];
            for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
            const double inv = nrm > 0 ? 1.0 / sqrt(nrm) : 1.0;
            for (int i = lane; i < n; i += 32) zv[i] *= inv;
            __syncwarp();
        }
        for (int i = lane; i < n; i += 32) {
            ZV(k, i) = zv[i];
            Z[i + (long)k * ldz] = make_double2(zv[i], 0.0);
        }
        __syncwarp();
    }
#undef ZV
}

// ------------------------------------------------------------------ back-transformation
// Z = Q z with Q = H_0 ... H_{n-2}, applied in blocks of IB reflectors from the last block
// to the first: Q_b = H_j0 ... H_j1-1 = I - V_b T_b V_b^H (compact WY form, T_b upper
// triangular), Z <- Z - V_b (T_b (V_b^H Z)).  T_b^-1 = strictly upper part of V_b^H V_b plus
// diag(1 / tau) (Joffrain, Low, Quintana-Orti, van de Geijn and Van Zee, 2006), so T_b^H is
// the inverse of a lower triangular matrix and comes from the kernel of the triangular
// solves.  A reflector with tau = 0 (H = I) gets a zero column and the diagonal entry 1.
// (Blocks of 32 with a column recurrence for T, and V_b^H V_b from warp-wide dot products on
// the FP64 units, took 9.2 ms at n = 816, m = 272.)

// V[:, j] <- 0 where tau_j = 0
__global__ void wy_zero_kernel(int n, double2* V, const double2* tau) {
    const int j = blockIdx.x;
    if (tau[j].x != 0.0 || tau[j].y != 0.0) return;
    for (int r = threadIdx.x; r < n; r += blockDim.x) V[r + (long)j * n] = make_double2(0.0, 0.0);
}
// M (lower, ld IB): strictly lower part of G = V_b^H V_b (which is the conjugate transpose of
// its strictly upper part), diagonal 1 / conj(tau) scaled to 1: row r of M times conj(tau_r)
// keeps tri_inv_kernel's real unit diagonal; the inverse's columns are scaled back in wy_scale
__global__ void wy_m_kernel(int nbk, double2* G, const double2* tau) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nbk * nbk) return;
    const int r = t % nbk, c = t / nbk;
    double2 tr = zconj(tau[r]);
    if (tr.x == 0.0 && tr.y == 0.0) tr = make_double2(1.0, 0.0);
    double2* g = G + r + (long)c * IB;
    *g = r > c ? cmul(tr, *g) : make_double2(r == c ? 1.0 : 0.0, 0.0);
}
// rows of X (b x m): X[r] *= tau_r (1 where tau = 0)
__global__ void wy_scale_kernel(int b, int m, double2* X, const double2* tau) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)b * m) return;
    const double2 tr = tau[t % b];
    if (tr.x == 0.0 && tr.y == 0.0) return;
    X[t] = cmul(X[t], tr);
}

inline int cdiv(long a, long b) { return (int)((a + b - 1) / b); }

// C(m, n) = alpha sum_z P(z, n, m) + beta C(m, n): 32 outputs per block, eight groups of
// consecutive z added in order (deterministic)
__global__ void __launch_bounds__(256) gemm_sum_kernel(int M, int N, int splits, const double2* P, double alpha,
                                                       double beta, OzDst C, int lower) {
    __shared__ double2 sh[8][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long total = (long)M * N, t = blockIdx.x * 32l + lane;
    const int m = (int)(t % M), n = (int)(t / M);
    const bool live = t < total && !(lower && (m / TB + 1) * TB <= (n / TB) * TB);  // (a tile the GEMM skipped)
    const int per = (splits + 7) / 8, z1 = min(splits, (w + 1) * per);
    double2 s = make_double2(0.0, 0.0);
    if (live)
#pragma unroll 4
        for (int z = w * per; z < z1; ++z) s = cadd(s, P[(size_t)z * total + t]);
    sh[w][lane] = s;
    __syncthreads();
    if (w || !live) return;
    for (int i = 1; i < 8; ++i) s = cadd(s, sh[i][lane]);
    double2* c = C.C + (C.mmap ? (long)C.mmap[m] : (long)m) * C.cm + (C.nmap ? (long)C.nmap[n] : (long)n) * C.cn;
    double2 o = make_double2(alpha * s.x, alpha * s.y);
    if (beta != 0.0) {
        o.x += beta * c->x;
        o.y += beta * c->y;
    }
    *c = o;
}

}  // namespace

// ------------------------------------------------------------------ host side
// C(m, n) = alpha sum_k a(m, k) b(k, n) + beta C(m, n).  From 6e7 flops on (and 64 k: the
// digit sums come out once per 64 k) on the tensor cores (fs_oz.cu): the FMA GEMM takes
// 90 us and more there, the digit form 60 to 90 us, all its passes included, and from
// 1e9 flops on a tenth.  Below that on the FP64 units; K is split over the grid's z
// dimension while there are fewer than four blocks per SM, into partial sums that a second
// kernel adds in a fixed order (deterministic).
void dense_gemm_mat(fs_ctx* c, int M, int N, int K, double alpha, const OzMat& A, const OzMat& B, double beta,
                    const OzDst& C, int table, int lower) {
    if (M <= 0 || N <= 0) return;
    K = std::max(K, 0);
    if (!lower && oz_worth(M, N, K) && oz_gemm(c, M, N, K, A, B, C, alpha, beta, table)) return;
    const int tiles = cdiv(M, TB) * cdiv(N, TB);
    int splits = 1;
    if (tiles < 4 * 152) splits = std::min(std::max(1, 4 * 152 / tiles), std::max(1, K / (2 * TK)));
    const int kc = std::max(1, cdiv(cdiv(K, splits), TK)) * TK;
    splits = std::max(1, cdiv(K, kc));
    double2* P = nullptr;
    if (splits > 1) {
        c->dense.gpart.ensure((size_t)splits * M * N * sizeof(double2));
        P = c->dense.gpart.as<double2>();
    }
    for (int y0 = 0; y0 < N; y0 += 65535 * TB) {  // one pass but for a very long N
        OzMat b = B;
        OzDst d = C;
        const int ny = std::min(N - y0, 65535 * TB);
        if (y0) {
            if (b.rp) b.rp += y0;
            else if (b.map) b.map += y0;
            else b.X += (long)y0 * b.sr;
            if (d.nmap) d.nmap += y0; else d.C += (long)y0 * d.cn;
        }
        zgemm_kernel<<<dim3(cdiv(M, TB), cdiv(ny, TB), splits), TB * TB, 0, c->stream>>>(M, ny, K, alpha, A, b, beta, d,
                                                                                      P, kc, lower);
        if (P)
            gemm_sum_kernel<<<cdiv((long)M * ny, 32), 256, 0, c->stream>>>(M, ny, splits, P, alpha, beta, d, lower);
    }
    FS_CUDA(cudaGetLastError());
}

namespace {
OzMat op_a(int op, const double2* A, int lda) { return OzMat{A, op == 0 ? 1l : (long)lda, op == 0 ? (long)lda : 1l, op == 1}; }
OzMat op_b(int op, const double2* B, int ldb) { return OzMat{B, op == 0 ? (long)ldb : 1l, op == 0 ? 1l : (long)ldb, op == 1}; }
}  // namespace

// C = alpha op(A) op(B) + beta C (column-major)
void dense_gemm(fs_ctx* c, int opA, int opB, int M, int N, int K, double alpha, const double2* A, int lda,
                const double2* B, int ldb, double beta, double2* C, int ldc) {
    dense_gemm_mat(c, M, N, K, alpha, op_a(opA, A, lda), op_b(opB, B, ldb), beta, OzDst{C, 1, ldc}, 0, 0);
}

// Cholesky of the lower triangle of A (n x n, ld lda); squared pivots to piv (device, may be
// null); info (device int, zeroed here): 0, or the first failing column + 1 as LAPACK's.
// Blocks of 32 within panels of PB columns; what a panel leaves to the columns beyond it is
// one product of PB k (on the tensor cores from 6e7 flops on).
static void potrf_async(fs_ctx* c, int n, double2* A, int lda, double* piv, int* info) {
    ProfScope ps(c, KS_SUB_POTRF, 0.0, 8.0 * n * (double)n * n / 3.0);
    constexpr int PB = 128;
    FS_CUDA(cudaMemsetAsync(info, 0, sizeof(int), c->stream));
    for (int p0 = 0; p0 < n; p0 += PB) {
        const int pe = std::min(n, p0 + PB);
        for (int j0 = p0; j0 < pe; j0 += NBLK) {
            const int b = std::min(NBLK, pe - j0);
            potrf_diag_kernel<<<1, PD_THREADS, 0, c->stream>>>(A, lda, j0, b, piv, info);
            const int rest = n - j0 - b;
            if (rest <= 0) continue;
            potrf_panel_kernel<<<cdiv((long)rest * 32, 128), 128, 0, c->stream>>>(A, lda, n, j0, b);
            // the panel's own remaining columns (lower triangle; the upper one is never read)
            const int own = pe - j0 - b;
            const double2* pan = A + j0 + b + (long)j0 * lda;
            if (own > 0)
                dense_gemm_mat(c, rest, own, b, -1.0, op_a(0, pan, lda), op_b(1, pan, lda), 1.0,
                               OzDst{A + j0 + b + (long)(j0 + b) * lda, 1, lda}, 0, 1);
        }
        const int rest = n - pe;
        if (rest > 0) {
            const double2* pan = A + pe + (long)p0 * lda;
            const bool big = oz_worth(rest, rest, pe - p0);
            dense_gemm_mat(c, rest, rest, pe - p0, -1.0, op_a(0, pan, lda), op_b(1, pan, lda), 1.0,
                           OzDst{A + pe + (long)pe * lda, 1, lda}, 0, big ? 0 : 1);
        }
    }
    FS_CUDA(cudaGetLastError());
}

// The same; returns the info.  Synchronises the context's stream.
int dense_potrf(fs_ctx* c, int n, double2* A, int lda, double* piv) {
    DenseWork& D = c->dense;
    D.info.ensure(2 * sizeof(int));
    potrf_async(c, n, A, lda, piv, D.info.as<int>());
    int h = 0;
    FS_CUDA(cudaMemcpyAsync(&h, D.info.p, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    ctx_check_errflag(c);  // (synchronises; before the info of a product that gave up is taken for one)
    return h;
}

// Inverses of the diagonal blocks of L (lower n x n) for the following dense_trsm calls with the same L
static void tri_inverses(fs_ctx* c, int n, const double2* L, int lda) {
    DenseWork& D = c->dense;
    D.linv.ensure((size_t)cdiv(n, IB) * IB * IB * sizeof(double2));
    tri_inv_kernel<<<cdiv((long)cdiv(n, IB) * IB, 4), 128, 0, c->stream>>>(L, lda, n, D.linv.as<double2>());
    FS_CUDA(cudaGetLastError());
}

// B <- L^-1 B (conj = 0) or L^-H B (conj = 1); L lower n x n (ld lda), B n x ncols (ld ldb).
// Blocks of IB rows: x_b = inv(L_bb) b_b, then the rest of B minus its product with x_b.
// fresh = false: the inverses of the last call's L are the ones of this L.
// The products are as exact as the rows of L are evenly scaled (see equil_scale_kernel): callers
// pass the factor of a matrix whose diagonal entries are of one size.
void dense_trsm(fs_ctx* c, int conj, int n, int ncols, const double2* L, int lda, double2* B, int ldb, bool fresh) {
    if (n <= 0 || ncols <= 0) return;
    ProfScope ps(c, KS_SUB_TRSM, 0.0, 4.0 * n * (double)n * ncols);
    if (fresh) tri_inverses(c, n, L, lda);
    DenseWork& D = c->dense;
    D.xb.ensure((size_t)IB * ncols * sizeof(double2));
    double2* X = D.xb.as<double2>();
    const int nblk = cdiv(n, IB);
    for (int q = 0; q < nblk; ++q) {
        const int bi = conj ? nblk - 1 - q : q;
        const int j0 = bi * IB, b = std::min(IB, n - j0);
        dense_gemm(c, conj ? 1 : 0, 0, b, ncols, b, 1.0, D.linv.as<double2>() + (size_t)bi * IB * IB, IB, B + j0, ldb,
                   0.0, X, b);
        FS_CUDA(cudaMemcpy2DAsync(B + j0, ldb * sizeof(double2), X, b * sizeof(double2), b * sizeof(double2), ncols,
                                  cudaMemcpyDeviceToDevice, c->stream));
        if (!conj) {
            const int rest = n - j0 - b;
            dense_gemm(c, 0, 0, rest, ncols, b, -1.0, L + j0 + b + (long)j0 * lda, lda, X, b, 1.0, B + j0 + b, ldb);
        } else {
            // B[0:j0] -= (L[j0:j0+b, 0:j0])^H X_b
            dense_gemm(c, 1, 0, j0, ncols, b, -1.0, L + j0, lda, X, b, 1.0, B, ldb);
        }
    }
    FS_CUDA(cudaGetLastError());
}

void dense_conj_transpose(fs_ctx* c, int n, int m, const double2* A, int lda, double2* out, int ldo) {
    conj_transpose_kernel<<<cdiv((long)n * m, 256), 256, 0, c->stream>>>(n, m, A, lda, out, ldo);
    FS_CUDA(cudaGetLastError());
}

// The m lowest eigenpairs of the Hermitian A (n x n, ld n, destroyed): w[0..m)
// ascending (device), Z (n x m, ld ldz, device) orthonormal eigenvectors.
void dense_heev(fs_ctx* c, int n, double2* A, int m, double* w, double2* Z, int ldz) {
    if (n <= 0 || m <= 0) return;
    if (n > FS_DENSE_MAX_N) throw fs_error(FS_ERR_ARG, "dense eigensolve larger than " + std::to_string(FS_DENSE_MAX_N));
    DenseWork& D = c->dense;
    D.V.ensure((size_t)n * n * sizeof(double2));
    D.tau.ensure((size_t)n * sizeof(double2));
    D.d.ensure((size_t)n * sizeof(double));
    D.e.ensure((size_t)n * sizeof(double));
    D.e2.ensure((size_t)n * sizeof(double));
    D.Y.ensure((size_t)2 * n * n * sizeof(double2));  // a row of y and a row of columns per step
    D.z.ensure((size_t)n * m * sizeof(double));
    D.info3.ensure(5 * sizeof(double));
    D.ds.ensure((size_t)n * sizeof(double));
    int dev = 0, nsm = 0;
    FS_CUDA(cudaGetDevice(&dev));
    FS_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    // four warps up to n = 1024 (8 rows a thread), eight beyond
    const int ht = n <= 1024 ? 128 : 256;
    const void* hk = n <= 128    ? (const void*)hetrd_kernel<128, 1>
                     : n <= 256  ? (const void*)hetrd_kernel<128, 2>
                     : n <= 512  ? (const void*)hetrd_kernel<128, 4>
                     : n <= 1024 ? (const void*)hetrd_kernel<128, 8>
                                 : (const void*)hetrd_kernel<256, 8>;
    if (!D.attr_set) {
        for (const void* k : {(const void*)hetrd_kernel<128, 1>, (const void*)hetrd_kernel<128, 2>,
                              (const void*)hetrd_kernel<128, 4>, (const void*)hetrd_kernel<128, 8>,
                              (const void*)hetrd_kernel<256, 8>})
            FS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, HETRD_SMEM));
        FS_CUDA(cudaFuncSetAttribute((const void*)tri_invit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     8 * FS_DENSE_MAX_N * (int)sizeof(double)));
        D.attr_set = true;
    }
    // a block per column, at most one per SM; the columns in shared memory when they fit
    // (n <= 1296 on 152 SMs)
    const int nblocks = std::max(1, std::min(nsm, n - 1));
    const size_t vecs = (size_t)2 * n * sizeof(double2) + (size_t)cdiv(n, nblocks) * (ht / 32) * sizeof(double2);
    const size_t own = (size_t)cdiv(n, nblocks) * n * sizeof(double2);
    int in_smem = vecs + own <= (size_t)HETRD_SMEM;
    const size_t smem = vecs + (in_smem ? own : 0);
    {
    ProfScope ps_h(c, KS_SUB_HETRD, 0.0, 16.0 * n * (double)n * n / 3.0);
    hermitize_kernel<<<cdiv((long)n * n, 256), 256, 0, c->stream>>>(A, n);
    FS_CUDA(cudaMemsetAsync(D.Y.p, 0xff, (size_t)2 * n * n * sizeof(double2), c->stream));  // EMPTY
    FS_CUDA(cudaMemsetAsync(D.V.p, 0, (size_t)n * n * sizeof(double2), c->stream));
    {
        int nn = n;
        double2* Ap = A;
        double2* Vp = D.V.as<double2>();
        double2* tp = D.tau.as<double2>();
        double* dp = D.d.as<double>();
        double* ep = D.e.as<double>();
        double2* Yp = D.Y.as<double2>();
        double2* Cp = Yp + (size_t)n * n;
        int* errp = ctx_errflag(c);
        void* args[] = {&nn, &Ap, &Vp, &tp, &dp, &ep, &Yp, &Cp, &in_smem, &errp};
        FS_CUDA(cudaLaunchCooperativeKernel(hk, nblocks, ht, args, smem, c->stream));
    }
    if (n == 1) {
        // no reflector: T = A
        FS_CUDA(cudaMemsetAsync(D.tau.p, 0, sizeof(double2), c->stream));
    }
    }
    {
    ProfScope ps_t(c, KS_SUB_TRIEIG, 0.0, 0.0);
    tri_prep_kernel<<<1, 256, 0, c->stream>>>(D.d.as<double>(), D.e.as<double>(), D.ds.as<double>(),
                                              D.e2.as<double>(), n, D.info3.as<double>());
    tri_bisect_kernel<<<m, 32, 0, c->stream>>>(D.ds.as<double>(), D.e2.as<double>(), n, m, D.info3.as<double>(), w);
    tri_invit_kernel<<<m, 32, (size_t)8 * n * sizeof(double), c->stream>>>(D.d.as<double>(), D.e.as<double>(), n, m,
                                                                           w, D.info3.as<double>(), D.z.as<double>(),
                                                                           Z, ldz);
    FS_CUDA(cudaGetLastError());
    }
    if (n > 1) {
        ProfScope ps_b(c, KS_SUB_BACK, 0.0, 8.0 * n * (double)n * m);
        const int nref = n - 1, nblkr = cdiv(nref, IB);
        D.wyT.ensure((size_t)nblkr * IB * IB * sizeof(double2));
        D.linv.ensure((size_t)nblkr * IB * IB * sizeof(double2));
        D.wyW.ensure((size_t)IB * m * sizeof(double2));
        D.wyW2.ensure((size_t)IB * m * sizeof(double2));
        double2* W = D.wyW.as<double2>();
        double2* W2 = D.wyW2.as<double2>();
        double2* G = D.wyT.as<double2>();
        const double2* tau = D.tau.as<double2>();
        double2* V = D.V.as<double2>();
        wy_zero_kernel<<<nref, 128, 0, c->stream>>>(n, V, tau);
        for (int b = 0; b < nblkr; ++b) {
            const int j0 = b * IB, nbk = std::min(IB, nref - j0), r0 = j0 + 1;  // v_j0 starts at row j0 + 1
            const double2* Vb = V + r0 + (long)j0 * n;
            dense_gemm(c, 1, 0, nbk, nbk, n - r0, 1.0, Vb, n, Vb, n, 0.0, G + (size_t)b * IB * IB, IB);
            wy_m_kernel<<<cdiv((long)nbk * nbk, 256), 256, 0, c->stream>>>(nbk, G + (size_t)b * IB * IB, tau + j0);
            tri_inv_kernel<<<IB / 4, 128, 0, c->stream>>>(G + (size_t)b * IB * IB, IB, nbk,
                                                          D.linv.as<double2>() + (size_t)b * IB * IB);
        }
        for (int b = nblkr - 1; b >= 0; --b) {
            const int j0 = b * IB, nbk = std::min(IB, nref - j0), r0 = j0 + 1, rows = n - r0;
            const double2* Vb = V + r0 + (long)j0 * n;
            // T^H = inv(D M') with M' = conj(tau) M of unit diagonal: T^H = inv(M') conj(tau), T = tau inv(M')^H
            dense_gemm(c, 1, 0, nbk, m, rows, 1.0, Vb, n, Z + r0, ldz, 0.0, W, nbk);
            dense_gemm(c, 1, 0, nbk, m, nbk, 1.0, D.linv.as<double2>() + (size_t)b * IB * IB, IB, W, nbk, 0.0, W2, nbk);
            wy_scale_kernel<<<cdiv((long)nbk * m, 256), 256, 0, c->stream>>>(nbk, m, W2, tau + j0);
            dense_gemm(c, 0, 0, rows, m, nbk, -1.0, Vb, n, W2, nbk, 1.0, Z + r0, ldz);
        }
        FS_CUDA(cudaGetLastError());
    }
    // one Cholesky QR pass: the vectors of eigenvalues outside a common cluster are orthogonal
    // only to about eps ||T|| / gap; their Gram matrix is I + O(that), so Z <- Z L^-H with
    // Z^H Z = L L^H restores orthonormality to working precision (it mixes only nearly
    // degenerate vectors)
    if (m > 1) {
        D.qrG.ensure((size_t)m * m * sizeof(double2));
        D.qrT.ensure((size_t)m * n * sizeof(double2));
        double2* G = D.qrG.as<double2>();
        double2* T = D.qrT.as<double2>();
        dense_gemm(c, 1, 0, m, m, n, 1.0, Z, ldz, Z, ldz, 0.0, G, m);
        // (should the factorisation fail, Z stays as it is: decided on the device)
        D.info.ensure(2 * sizeof(int));
        int* info = D.info.as<int>() + 1;
        potrf_async(c, m, G, m, nullptr, info);
        dense_conj_transpose(c, n, m, Z, ldz, T, m);
        dense_trsm(c, 0, m, n, G, m, T, m, true);
        qr_back_kernel<<<cdiv((long)n * m, 256), 256, 0, c->stream>>>(n, m, T, Z, ldz, info);
        FS_CUDA(cudaGetLastError());
    }
}

// Generalised Hermitian problem GA x = lambda GB x (both n x n, ld n; GB positive
// definite): the m lowest pairs; eigenvectors (GB-orthonormal) overwrite GA's
// first m columns, eigenvalues to w.  GB is overwritten.
// Returns the Cholesky info (0 = success).
int dense_hegv(fs_ctx* c, int n, double2* GA, double2* GB, int m, double* w) {
    DenseWork& D = c->dense;
    // scaled where a product of the triangular solves goes to the tensor cores (n >= 315);
    // the FMA products do not need it, and its launches are 8 us of 300 to 2,000 there
    const bool scaled = oz_worth(std::max(std::min(n, IB), n - IB), n, std::min(n, IB));
    D.equil.ensure((size_t)2 * n * sizeof(double));
    const double* s = D.equil.as<double>();
    if (scaled) {
        equil_scale_kernel<<<cdiv(n, 256), 256, 0, c->stream>>>(GB, n, D.equil.as<double>());
        equil_sym_kernel<<<cdiv((long)n * n, 256), 256, 0, c->stream>>>(GA, GB, n, s);
        FS_CUDA(cudaGetLastError());
    }
    int info = dense_potrf(c, n, GB, n, nullptr);
    if (info != 0) return info;
    D.T.ensure((size_t)n * n * sizeof(double2));
    D.U.ensure((size_t)n * m * sizeof(double2));
    double2* T = D.T.as<double2>();
    // (dense_heev's own triangular solve replaces the kept inverses)
    dense_trsm(c, 0, n, n, GB, n, GA, n, true);        // L^-1 GA
    dense_conj_transpose(c, n, n, GA, n, T, n);         // (L^-1 GA)^H = GA L^-H
    dense_trsm(c, 0, n, n, GB, n, T, n, false);        // L^-1 GA L^-H
    dense_heev(c, n, T, m, w, D.U.as<double2>(), n);
    dense_trsm(c, 1, n, m, GB, n, D.U.as<double2>(), n, true);  // x = L^-H y
    if (scaled)
        equil_rows_kernel<<<cdiv((long)n * m, 256), 256, 0, c->stream>>>(D.U.as<double2>(), n, m, s, GA);
    else
        FS_CUDA(cudaMemcpyAsync(GA, D.U.p, (size_t)n * m * sizeof(double2), cudaMemcpyDeviceToDevice, c->stream));
    FS_CUDA(cudaGetLastError());
    return 0;
}

// ------------------------------------------------------------------ C ABI (checking the dense solvers)
extern "C" fs_status fs_dense_eigh(fs_ctx* c, int n, const void* A, const void* B, int m, double* w, void* Z) {
    if (!c) return FS_ERR_ARG;
    if (n <= 0 || n > FS_DENSE_MAX_N || m <= 0 || m > n || !A || !w || !Z) {
        c->err = "fs_dense_eigh: bad arguments";
        return FS_ERR_ARG;
    }
    return ctx_call(c, [&] {
        const size_t bytes = (size_t)n * n * sizeof(double2);
        dbuf dA, dB, dZ, dw;
        dA.alloc(bytes);
        dZ.alloc((size_t)n * m * sizeof(double2));
        dw.alloc((size_t)n * sizeof(double));
        FS_CUDA(cudaMemcpyAsync(dA.p, A, bytes, cudaMemcpyHostToDevice, c->stream));
        if (B) {
            dB.alloc(bytes);
            FS_CUDA(cudaMemcpyAsync(dB.p, B, bytes, cudaMemcpyHostToDevice, c->stream));
            const int info = dense_hegv(c, n, dA.as<double2>(), dB.as<double2>(), m, dw.as<double>());
            if (info != 0) throw fs_error(FS_ERR_NUMERIC, "fs_dense_eigh: B is not positive definite (column " +
                                                              std::to_string(info) + ")");
            FS_CUDA(cudaMemcpyAsync(dZ.p, dA.p, (size_t)n * m * sizeof(double2), cudaMemcpyDeviceToDevice,
                                    c->stream));
        } else {
            dense_heev(c, n, dA.as<double2>(), m, dw.as<double>(), dZ.as<double2>(), n);
        }
        FS_CUDA(cudaMemcpyAsync(w, dw.p, (size_t)m * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        FS_CUDA(cudaMemcpyAsync(Z, dZ.p, (size_t)n * m * sizeof(double2), cudaMemcpyDeviceToHost, c->stream));
        FS_CUDA(cudaStreamSynchronize(c->stream));
    });
}
