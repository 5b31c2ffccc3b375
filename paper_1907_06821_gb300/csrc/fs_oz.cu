// FP64 complex GEMM on the 5th-generation tensor cores, by error-free splitting
// (the scheme of Ozaki, Ogita, Oishi and Rump, 2012, in its fixed-point form).
//
//   C(m, n) = alpha sum_k opA(a(m, k)) opB(b(k, n)) + beta C(m, n)
//
// Each operand row (a over k for fixed m, b over k for fixed n) gets one power of
// two 2^E above its largest component; every component is rounded to a signed
// 56-bit fixed-point number x 2^(55 - E) and cut into seven signed 8-bit digits
// (most significant first).  Digits are exact in BF16, the product of two digits is
// at most 2^14, and a sum of 64 complex k over the at most 7 digit pairs (i, j)
// with i + j = d stays below 2^24: tcgen05.mma kind::f16 with FP32 accumulators
// computes the eight sums D_0 .. D_7 of that chunk without any rounding.  They are
// read out as integers and added to two 64-bit integers per output,
//     hi += D_0 2^16 + D_1 2^8 + D_2,   lo += D_3 2^24 + D_4 2^16 + D_5 2^8 + D_6 + D_7 / 2^8
// (the last rounded to an integer), and C = (hi 2^32 + lo) 2^(Ea + Eb - 62).
// The error is that of the cut, up to 2^-55 of the row maximum per component (2^(E - 56), and
// the maximum may be 2^(E - 1)); the digit pairs left out (i + j > 7) and the rounding of D_7 are
// below it.  So it is relative to (largest |a| of a row) x (largest |b| of a column), where an FMA
// chain's is relative to sum |a||b|: no larger for operands whose k contribute alike (Gram
// products, rotations, projections; with 28 MMAs a stage, without the pairs i + j = 7, it was 1.5
// to 8 times as large), larger where a and b are graded along k in opposite directions.  The
// triangular solves, where that can happen, work on scaled factors (fs_dense.cu).
//
// Why: GB300 does about 2 FP64 FMAs per clock and SM (0.65 TFLOP/s through a GEMM);
// 34 BF16 digit products at the tensor rate are some 50 times as fast.  What bounds
// it then: with few columns the digit images (28 bytes per complex element) from
// HBM; with many the MMAs and the formatting passes.  Measured: 272 x 272 x 193,673 in
// 7.6 ms (15 TFLOP/s, formatting included) against about 180 ms, relative error 1.4e-16
// against 0.5 to 1.2e-15; an FP64 H application of 16 bands of 193,673 plane waves with
// 2,048 projectors (table images kept) in 6.7 ms against 305 ms, 2.1 ms for each of its
// two products (11 GB of digits: 1.6 ms).
//
// Layout.  The complex product is carried by interleaved real rows: the A image of a
// row holds (re, im) pairs, the B image two rows per n, (re, -im) and (im, re) of b
// (or (re, im) and (im, -re) when a is conjugated).  An image stage (8 complex k)
// is the exact shared-memory image of the seven digit slices, K-major core matrices
// of 8 rows x 16 bytes, so one bulk copy moves it.
#include "fs_common.cuh"

#include <algorithm>
#include <cfloat>
#include <climits>

namespace {

constexpr int NS = 7;                         // digits of an operand
constexpr int ND = 8;                         // accumulators: digit pairs (i, j) by i + j
constexpr int OM = 128;                       // rows of a tile (UMMA M)
constexpr int ON2_MAX = 64;                   // UMMA N: two real rows per column of C
constexpr int OKC = 8;                        // complex k per stage (UMMA K = 16 reals)
constexpr int OCHAIN = 8;                     // stages per accumulation chain (64 complex k: exact)
constexpr int OA_SLICE = OM * 32;             // bytes of one digit slice of an A stage
constexpr int OA_STAGE = NS * OA_SLICE;
constexpr int O_THREADS = 320;
constexpr int O_SMEM_MAX = 232448;
constexpr int O_CTL = 256;
__host__ __device__ constexpr int O_COLS(int nq) { return nq == 1 ? 256 : 512; }  // tensor-memory columns
constexpr int O_STAGES_MAX = 8;
constexpr int E_MIN = -900;                   // exponent of an all-zero row (components below 2^-954 read as 0)
constexpr long long OZ_WAIT_LIMIT = 1ll << 28;

__device__ __forceinline__ uint32_t oz_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool oz_wait(uint64_t* bar, uint32_t parity) {
    const uint32_t a = oz_smem(bar);
    for (long long it = 0; it < OZ_WAIT_LIMIT; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void oz_init_bar(uint64_t* bar, int n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(oz_smem(bar)), "r"(n));
}
__device__ __forceinline__ void oz_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(oz_smem(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void oz_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(oz_smem(bar)) : "memory");
}
__device__ __forceinline__ void oz_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     oz_smem(dst)),
                 "l"(src), "r"(bytes), "r"(oz_smem(bar))
                 : "memory");
}
__device__ __forceinline__ void oz_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(oz_smem(bar))
                 : "memory");
}
__device__ __forceinline__ void oz_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void oz_ld8(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// byte offset of the 16-byte chunk (row, half) of a digit slice: two core matrices along K
__host__ __device__ __forceinline__ uint32_t oz_chunk(int row, int half) {
    return (uint32_t)((((row >> 3) * 2 + half) << 7) + ((row & 7) << 4));
}
__device__ __forceinline__ uint64_t oz_desc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)(128 >> 4) << 16;  // leading byte offset: next core matrix along K
    d |= (uint64_t)(256 >> 4) << 32;  // stride byte offset: next 8-row group
    d |= (uint64_t)1 << 46;
    return d;
}

// exponent E of a row from the bits of its largest magnitude.  Seven signed digits hold up to
// 0x7F7F7F7F7F7F7F = 0.49803 2^56, i.e. |x| <= 0.99607 2^E: a mantissa at the top of its range
// (six leading ones, |x| >= 0.992 of the next power) takes the next exponent
__device__ __forceinline__ int oz_exp(unsigned long long bits) {
    const int e = (int)(bits >> 52) - 1022 + (((bits >> 46) & 0x3f) == 0x3f ? 1 : 0);
    return e < E_MIN ? E_MIN : e;
}

// ---------------------------------------------------------------- row maxima
// An operand: element (r, k) = X[map(r) * sr + kmap(k) * sk] (maps may be null).
struct OzOp {
    const double2* X;
    long sr, sk;
    const int* map;
    const int* kmap;
    const double2* const* rp;  // rows, or k, by pointers
    const double2* const* kp;
    __device__ __forceinline__ const double2& at(int r, long k) const {
        if (rp) return rp[r][k * sk];
        if (kp) return kp[k][r * sr];
        return X[(map ? (long)map[r] : (long)r) * sr + (kmap ? (long)kmap[k] : k) * sk];
    }
};

// largest magnitude (as bits) of every row over k in [0, K).  sk = 1: a warp walks along k;
// else a thread per row (consecutive rows are consecutive in memory).
__global__ void oz_max_kernel(OzOp op, int R, int K, int kper, unsigned long long* __restrict__ out) {
    const int k0 = blockIdx.y * kper, k1 = min(K, k0 + kper);
    if (op.sk == 1) {
        const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (r >= R) return;
        unsigned long long m = 0;
#pragma unroll 4
        for (int k = k0 + lane; k < k1; k += 32) {
            const double2 v = op.at(r, k);
            m = max(m, max((unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull,
                           (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull));
        }
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) atomicMax(out + r, m);
    } else {
        const int r = blockIdx.x * blockDim.x + threadIdx.x;
        if (r >= R) return;
        unsigned long long m = 0;
#pragma unroll 4
        for (int k = k0; k < k1; ++k) {
            const double2 v = op.at(r, k);
            m = max(m, max((unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull,
                           (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull));
        }
        atomicMax(out + r, m);
    }
}

// ---------------------------------------------------------------- digit images
// biased digits of x: byte s of the result is digit s + 128 (s = 0 least significant)
__device__ __forceinline__ unsigned long long oz_digits(double x, double scale) {
    return (unsigned long long)__double2ll_rn(x * scale) + 0x0080808080808080ull;
}
// digit s of two numbers as two BF16 values (lo half: p, hi half: q), exact
__device__ __forceinline__ uint32_t oz_pair(unsigned long long p, unsigned long long q, int s) {
    const float fp = __uint_as_float(0x4B000000u | (uint32_t)((p >> (8 * s)) & 0xff)) - 8388736.0f;
    const float fq = __uint_as_float(0x4B000000u | (uint32_t)((q >> (8 * s)) & 0xff)) - 8388736.0f;
    return __byte_perm(__float_as_uint(fp), __float_as_uint(fq), 0x7632);
}

// The 16-byte chunk ch (4 complex k) of local row lr (operand row r) in every slice.
//   BSIDE = false: A image, tiles of 128 rows
//   BSIDE = true : B image, tiles of tr = N2 / 2 operand rows, two image rows each;
//                  conja / conjb: conjugated A and B of the product
template <bool BSIDE>
__device__ __forceinline__ void oz_put(const OzOp& op, int lr, int r, int R, long ch, int K, int tr, int kb0, int nkb,
                                       int conja, int conjb, double scale, unsigned char* __restrict__ out) {
    const uint32_t slice = BSIDE ? (uint32_t)tr * 64 : (uint32_t)OA_SLICE;
    unsigned long long d[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) d[q] = 0x0080808080808080ull;  // digits of 0
    if (r < R) {
        const long k = (long)kb0 * OKC + 4 * ch;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (k + q < K) {
                const double2 v = op.at(r, k + q);
                d[2 * q] = oz_digits(v.x, scale);
                d[2 * q + 1] = oz_digits(v.y, scale);
            }
    }
    const long kb = ch >> 1;
    const int half = (int)(ch & 1);
    if (!BSIDE) {
        unsigned char* st = out + ((long)(lr / OM) * nkb + kb) * OA_STAGE + oz_chunk(lr % OM, half);
#pragma unroll
        for (int s = 0; s < NS; ++s)
            *reinterpret_cast<uint4*>(st + s * OA_SLICE) =
                make_uint4(oz_pair(d[0], d[1], NS - 1 - s), oz_pair(d[2], d[3], NS - 1 - s),
                           oz_pair(d[4], d[5], NS - 1 - s), oz_pair(d[6], d[7], NS - 1 - s));
    } else {
        // b' = conjb ? conj(b) : b; rows (b'r, -b'i), (b'i, b'r), or with conja (b'r, b'i), (b'i, -b'r)
        const uint32_t s0 = (conja != 0) == (conjb != 0) ? 0x80000000u : 0u;  // sign of the im half, first row
        const uint32_t s1l = conjb ? 0x00008000u : 0u;                        // sign of im, second row
        const uint32_t s1h = conja ? 0x80000000u : 0u;                        // sign of re, second row
        const int tile = lr / tr, j = lr - tile * tr;
        unsigned char* st = out + ((long)tile * nkb + kb) * ((long)NS * slice);
        const uint32_t o0 = oz_chunk(2 * j, half);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            uint32_t a[4], b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t p = oz_pair(d[2 * q], d[2 * q + 1], NS - 1 - s);  // (re, im)
                a[q] = p ^ s0;
                b[q] = __byte_perm(p, p, 0x1032) ^ (s1l | s1h);                   // (im, re)
            }
            unsigned char* sl = st + (long)s * slice;
            *reinterpret_cast<uint4*>(sl + o0) = make_uint4(a[0], a[1], a[2], a[3]);
            *reinterpret_cast<uint4*>(sl + o0 + 16) = make_uint4(b[0], b[1], b[2], b[3]);
        }
    }
}

__device__ __forceinline__ double oz_scale(unsigned long long bits) {
    return __longlong_as_double((long long)(55 - oz_exp(bits) + 1023) << 52);
}

// Rows r0 .., stages [kb0, kb0 + nkb) of the operand as local stages 0 .. nkb, by known maxima
template <bool BSIDE>
__global__ void oz_fmt_kernel(OzOp op, int r0, int R, int K, int rows, int tr, int kb0, int nkb, int conja, int conjb,
                              const unsigned long long* __restrict__ rmax, unsigned char* __restrict__ out) {
    const bool kcont = op.sk == 1;
    const long nch = 2l * nkb;  // chunks of 4 complex k per row
    const long total = kcont ? (long)(rows / 8) * ((nch + 3) / 4) * 32 : (long)rows * nch;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        int lr;   // local row
        long ch;  // local chunk
        if (kcont) {  // 8 rows x 4 chunks per warp (rows is a multiple of 8; chunk groups of 4)
            const int lane = (int)(t & 31);
            const long w = t >> 5, ncg = (nch + 3) / 4;
            lr = (int)(w / ncg) * 8 + (lane & 7);
            ch = (w % ncg) * 4 + (lane >> 3);
            if (ch >= nch) continue;
        } else {
            lr = (int)(t % rows);
            ch = t / rows;
        }
        const int r = r0 + lr;
        oz_put<BSIDE>(op, lr, r, R, ch, K, tr, kb0, nkb, conja, conjb, r < R ? oz_scale(rmax[r]) : 0.0, out);
    }
}

// Maxima and images in one launch, all K.  Rows along k (short ones): 8 rows per block, a warp
// finds a row's maximum.  Rows contiguous in memory: 32 rows per block, a warp takes every
// eighth k, then every eighth chunk.  (Three launches an operand made a small product 60 us.)
template <bool BSIDE>
__global__ void __launch_bounds__(256) oz_maxfmt_kernel(OzOp op, int r0, int R, int K, int rows, int tr, int nkb,
                                                        int conja, int conjb, unsigned long long* __restrict__ rmax,
                                                        unsigned char* __restrict__ out) {
    __shared__ unsigned long long part[8][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto mag = [&](int r, int k) {
        const double2 v = op.at(r, k);
        return max((unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull,
                   (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull);
    };
    unsigned long long m = 0;
    if (op.sk == 1) {
        const int lr0 = blockIdx.x * 8, r = r0 + lr0 + w;
        if (r < R)
#pragma unroll 4
            for (int k = lane; k < K; k += 32) m = max(m, mag(r, k));
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) {
            part[0][w] = m;
            if (r < R) rmax[r] = m;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < 16 * nkb; t += 256) {
            const int lr = lr0 + (t & 7);
            oz_put<BSIDE>(op, lr, r0 + lr, R, t >> 3, K, tr, 0, nkb, conja, conjb, oz_scale(part[0][t & 7]), out);
        }
    } else {
        const int lr = blockIdx.x * 32 + lane, r = r0 + lr;
        if (r < R)
#pragma unroll 4
            for (int k = w; k < K; k += 8) m = max(m, mag(r, k));
        part[w][lane] = m;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) m = max(m, part[i][lane]);
        if (w == 0 && r < R) rmax[r] = m;
        const double s = oz_scale(m);
        if (lr < rows)
            for (int ch = w; ch < 2 * nkb; ch += 8)
                oz_put<BSIDE>(op, lr, r, R, ch, K, tr, 0, nkb, conja, conjb, s, out);
    }
}

// ---------------------------------------------------------------- the GEMM
struct OzOut {
    double2* C;        // element (m, n) at C[mmap(m) * cm + nmap(n) * cn]
    long cm, cn;
    const int *mmap, *nmap;
    double alpha, beta;
    double2* part;     // split K: partial (z, n, m) at part[(z * N + n) * M + m] (raw sums), else null
};

// grid (jtiles, itiles, splits).  Warp 0 copies the stages, warp 1 issues the MMAs of
// each (34 digit pairs i + j <= 7 into accumulator i + j), warps 2-9 drain the eight
// accumulators of a chain (thread: row 32 (warp & 3) + lane, half of the columns).
// Two accumulator sets when 16 N2 <= 512 columns of tensor memory, else one.
// NQ: groups of 8 accumulator columns per drain thread (N2 <= 16 NQ).  With one group (at most
// eight columns of C) two blocks fit on an SM (registers, tensor memory, half the ring each), so
// that one's start and epilogue run under the other's copies.
template <int NQ>
__global__ void __launch_bounds__(O_THREADS, NQ == 1 ? 2 : 1)
oz_gemm_kernel(int M, int N, int m0, int N2, int nkb, int kbs, int nst, const unsigned char* __restrict__ Af,
               long a_stride, long a_kb0, const unsigned char* __restrict__ Bf, const unsigned long long* __restrict__ ma,
               const unsigned long long* __restrict__ mb, OzOut o, int z0, int* errflag) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t bslice = (uint32_t)N2 * 32, bstage = NS * bslice, sbytes = OA_STAGE + bstage;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)nst * sbytes);
    uint64_t* empty = full + nst;
    uint64_t* accf = empty + nst;
    uint64_t* acce = accf + 2;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(acce + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            oz_init_bar(&full[s], 1);
            oz_init_bar(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            oz_init_bar(&accf[b], 1);
            oz_init_bar(&acce[b], 8);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(oz_smem(tslot)), "r"(O_COLS(NQ)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;
    const int jt = blockIdx.x, it = blockIdx.y, z = blockIdx.z;
    const int kb0 = z * kbs, nk = min(nkb, kb0 + kbs) - kb0;
    const int nbuf = 2 * ND * N2 <= O_COLS(NQ) ? 2 : 1;
    const int nchain = (nk + OCHAIN - 1) / OCHAIN;
    const unsigned char* a = Af + ((long)it * a_stride + a_kb0 + kb0) * OA_STAGE;
    const unsigned char* b = Bf + ((long)jt * nkb + kb0) * (long)bstage;
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            int last = -1;
            for (int kb = 0; kb < nk; ++kb) {
                const int s = kb % nst;
                if (kb >= nst && !oz_wait(&empty[s], ((kb / nst) - 1) & 1)) {
                    ok = false;
                    break;
                }
                unsigned char* st = smem + (size_t)s * sbytes;
                oz_expect(&full[s], sbytes);
                oz_copy(st, a + (long)kb * OA_STAGE, OA_STAGE, &full[s]);
                oz_copy(st + OA_STAGE, b + (long)kb * bstage, bstage, &full[s]);
                last = kb;
            }
            // every copy issued has landed before the block can exit
            for (int kb = max(0, last - nst + 1); kb <= last; ++kb)
                if (!oz_wait(&full[kb % nst], (kb / nst) & 1)) ok = false;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // kind::f16, BF16 A and B, FP32 D, K-major both
            // (the number of columns is added per MMA)
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(OM >> 4) << 24);
            const int per = 256 / N2;  // digits of B per MMA
            int last = -1;
            for (int kb = 0; kb < nk; ++kb) {
                const int s = kb % nst, ch = kb / OCHAIN, buf = ch % nbuf;
                const bool first = kb % OCHAIN == 0;
                if (!oz_wait(&full[s], (kb / nst) & 1)) {
                    ok = false;
                    break;
                }
                if (first && ch >= nbuf && !oz_wait(&acce[buf], ((ch / nbuf) - 1) & 1)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = oz_smem(smem + (size_t)s * sbytes);
                const uint64_t ad = oz_desc(base), bd = oz_desc(base + OA_STAGE);
                const uint32_t d0 = tmem + (uint32_t)(buf * ND * N2);
                // digit i of A times digits j0 .. j1 of B at once: the slices of B follow one
                // another in shared memory as the accumulators i + j do in tensor memory, so
                // they are one operand of (j1 - j0) N2 <= 256 rows.  (One MMA per pair read A
                // from shared memory 34 times a stage and ran below the full rate at N <= 64.)
#pragma unroll
                for (int i = 0; i < NS; ++i) {
                    const int nj = i == 0 ? NS : ND - i;
                    for (int j0 = 0, j1; j0 < nj; j0 = j1) {
                        j1 = min(nj, j0 + per);
                        // accumulator 7 starts with (1, 6), the others with i = 0
                        if (first && i == 1 && j0 < NS - 1) j1 = min(j1, NS - 1);
                        const uint32_t acc = first && (i == 0 || (i == 1 && j0 == NS - 1)) ? 0u : 1u;
                        oz_mma(d0 + (uint32_t)((i + j0) * N2), ad + (uint64_t)((i * OA_SLICE) >> 4),
                               bd + (uint64_t)((j0 * bslice) >> 4), idesc + ((uint32_t)((j1 - j0) * (N2 >> 3)) << 17),
                               acc);
                    }
                }
                oz_commit(&empty[s]);
                if (kb % OCHAIN == OCHAIN - 1 || kb == nk - 1) oz_commit(&accf[buf]);
                last = kb;
            }
            // the MMAs issued have completed before tensor memory is released
            if (last >= 0 && !oz_wait(&empty[last % nst], (last / nst) & 1)) ok = false;
        }
    } else {
        const int q = warp & 3, h = (warp - 2) >> 2;
        const int nq = N2 >> 4;  // groups of 8 accumulator columns of this half
        long long hi[NQ][8], lo[NQ][8];
#pragma unroll
        for (int g = 0; g < NQ; ++g)
#pragma unroll
            for (int e = 0; e < 8; ++e) hi[g][e] = lo[g][e] = 0;
        for (int ch = 0; ch < nchain; ++ch) {
            const int buf = ch % nbuf;
            // every lane polls; the vote keeps the warp together if one gives up
            if (!__all_sync(0xffffffffu, oz_wait(&accf[buf], (ch / nbuf) & 1))) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t t0 = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * ND * N2 + h * (N2 >> 1));
#pragma unroll
            for (int g = 0; g < NQ; ++g)
                if (g < nq) {  // warp-uniform
                    uint32_t r[ND][8];
#pragma unroll
                    for (int d = 0; d < ND; ++d) oz_ld8(t0 + (uint32_t)(d * N2 + 8 * g), r[d]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        int v[ND];
#pragma unroll
                        for (int d = 0; d < ND; ++d) v[d] = __float2int_rn(__uint_as_float(r[d][e]));
                        hi[g][e] += (long long)v[0] * 65536 + ((long long)v[1] * 256 + v[2]);
                        lo[g][e] += ((long long)v[3] * 65536 + ((long long)v[4] * 256 + v[5])) * 256 +
                                    (v[6] + ((v[7] + 128) >> 8));
                    }
                }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) oz_arrive(&acce[buf]);
        }
        const int ml = it * OM + 32 * q + lane, m = m0 + ml;
        if (ok && m < M) {
            const unsigned long long am = ma[m];
            const int ea = oz_exp(am);
#pragma unroll
            for (int g = 0; g < NQ; ++g)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int jj = h * (N2 >> 2) + 4 * g + e, n = jt * (N2 >> 1) + jj;
                    if (g < nq && n < N) {
                        const unsigned long long bm = mb[n];
                        // the power of two in two factors (each within the range of a double)
                        const int ex = ea + oz_exp(bm) - 62, e1 = ex / 2, e2 = ex - e1;
                        const double f1 = __longlong_as_double((long long)(e1 + 1023) << 52);
                        const double f2 = __longlong_as_double((long long)(e2 + 1023) << 52);
                        double re = fma((double)hi[g][2 * e], 4294967296.0, (double)lo[g][2 * e]) * f1 * f2;
                        double im = fma((double)hi[g][2 * e + 1], 4294967296.0, (double)lo[g][2 * e + 1]) * f1 * f2;
                        // a row holding Inf or NaN has no digits: its products are not numbers
                        if (am >= 0x7ff0000000000000ull || bm >= 0x7ff0000000000000ull)
                            re = im = __longlong_as_double(0x7ff8000000000000ll);
                        if (o.part) {
                            o.part[((long)(z0 + z) * N + n) * M + m] = make_double2(re, im);
                        } else {
                            double2* c = o.C + (o.mmap ? (long)o.mmap[m] : (long)m) * o.cm +
                                         (o.nmap ? (long)o.nmap[n] : (long)n) * o.cn;
                            double2 v = make_double2(o.alpha * re, o.alpha * im);
                            if (o.beta != 0.0) {
                                const double2 old = *c;
                                v.x += o.beta * old.x;
                                v.y += o.beta * old.y;
                            }
                            *c = v;
                        }
                    }
                }
        }
    }
    if (!ok) *(volatile int*)errflag = 1;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(O_COLS(NQ)));
}

// C(m, n) = alpha sum_z part(z, n, m) + beta C(m, n): 32 outputs per block, eight groups of
// consecutive z added in order (deterministic)
__global__ void __launch_bounds__(256) oz_sum_kernel(int M, int N, int splits, OzOut o) {
    __shared__ double2 sh[8][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long total = (long)M * N, t = blockIdx.x * 32l + lane;
    const int per = (splits + 7) / 8, z1 = min(splits, (w + 1) * per);
    double2 s = make_double2(0.0, 0.0);
    if (t < total)
#pragma unroll 4
        for (int z = w * per; z < z1; ++z) s = cadd(s, o.part[(long)z * total + t]);
    sh[w][lane] = s;
    __syncthreads();
    if (w || t >= total) return;
    for (int i = 1; i < 8; ++i) s = cadd(s, sh[i][lane]);
    const long n = t / M, m = t - n * M;
    double2* c = o.C + (o.mmap ? (long)o.mmap[m] : m) * o.cm + (o.nmap ? (long)o.nmap[n] : n) * o.cn;
    double2 v = make_double2(o.alpha * s.x, o.alpha * s.y);
    if (o.beta != 0.0) {
        v.x += o.beta * c->x;
        v.y += o.beta * c->y;
    }
    *c = v;
}

inline int cdiv_(long a, long b) { return (int)((a + b - 1) / b); }

void row_max(fs_ctx* c, const OzOp& op, int R, int K, unsigned long long* out) {
    FS_CUDA(cudaMemsetAsync(out, 0, (size_t)R * sizeof(unsigned long long), c->stream));
    const int bx = op.sk == 1 ? cdiv_(R, 8) : cdiv_(R, 256);
    const int by = std::max(1, std::min(cdiv_(K, 64), 152 * 8 / std::max(1, bx)));
    oz_max_kernel<<<dim3(bx, std::min(by, 65535)), 256, 0, c->stream>>>(op, R, K, cdiv_(K, by), out);
}

template <bool BSIDE>
void maxfmt(fs_ctx* c, const OzOp& op, int r0, int R, int K, int rows, int tr, int nkb, int conja, int conjb,
            unsigned long long* rmax, unsigned char* out) {
    oz_maxfmt_kernel<BSIDE><<<op.sk == 1 ? rows / 8 : cdiv_(rows, 32), 256, 0, c->stream>>>(
        op, r0, R, K, rows, tr, nkb, conja, conjb, rmax, out);
}

template <bool BSIDE>
void fmt(fs_ctx* c, const OzOp& op, int r0, int R, int K, int rows, int tr, int kb0, int nkb, int conja, int conjb,
         const unsigned long long* rmax, unsigned char* out) {
    // whole warps: 8 rows x 4 chunks
    const long thr = op.sk == 1 ? (long)(rows / 8) * ((2l * nkb + 3) / 4) * 32 : (long)rows * 2 * nkb;
    oz_fmt_kernel<BSIDE><<<(int)std::min<long>(152 * 16, (thr + 255) / 256), 256, 0, c->stream>>>(
        op, r0, R, K, rows, tr, kb0, nkb, conja, conjb, rmax, out);
}

}  // namespace

// sizes from which the tensor-core form is taken (see dense_gemm_mat)
bool oz_worth(int M, int N, int K) { return 8.0 * M * N * (double)K >= 6e7 && K >= 64 && std::max(M, N) >= 32; }

// Whether the context may keep a digit image of `bytes` of its projector table: small ones always,
// others while they take at most an eighth of the memory then free, so that the library's and the
// program's other buffers find the room they had.
static bool image_fits(size_t bytes) {
    if (bytes <= 256ull << 20) return true;
    if (bytes > FS_TABLE_FMT_MAX_BYTES) return false;
    size_t avail = 0, total = 0;
    FS_CUDA(cudaMemGetInfo(&avail, &total));
    return bytes <= avail / 8;
}

// C(m, n) = alpha sum_k a(m, k) b(k, n) + beta C(m, n) on the tensor cores (header of this file).
// Of the two ways round (either operand as the 128-row side) the one with less padded work is taken.
// Every buffer is allocated before the first launch; where the images do not fit, they are made in
// smaller chunks, and false is returned if that does not help either.
bool oz_gemm(fs_ctx* c, int M, int N, int K, const OzMat& Am, const OzMat& Bm, const OzDst& Cd, double alpha,
             double beta, int table) {
    auto cost = [](int m, int n) {  // tiles x cycles of an MMA: shared-memory reads of both operands
        const int jt = cdiv_(n, ON2_MAX / 2), n2 = 2 * cdiv_(cdiv_(n, jt), 8) * 8;
        return (double)cdiv_(m, OM) * jt * (32 + n2 / 4);
    };
    if (!table && cost(N, M) < cost(M, N))
        return oz_gemm(c, N, M, K, Bm, Am, OzDst{Cd.C, Cd.cn, Cd.cm, Cd.nmap, Cd.mmap}, alpha, beta, -1);
    table = std::max(table, 0);
    const int conja = Am.conj, conjb = Bm.conj;
    smem_limit(c->oz_limit, O_SMEM_MAX,
               {(const void*)oz_gemm_kernel<1>, (const void*)oz_gemm_kernel<2>, (const void*)oz_gemm_kernel<4>});
    OzWork& W = c->oz;
    struct Busy {
        bool& b;
        explicit Busy(bool& x) : b(x) { b = true; }
        ~Busy() { b = false; }
    } busy(W.busy);
    const OzOp a{Am.X, Am.sr, Am.sk, Am.map, Am.kmap, Am.rp, Am.kp},
        b{Bm.X, Bm.sr, Bm.sk, Bm.map, Bm.kmap, Bm.rp, Bm.kp};
    const int nkb = cdiv_(K, OKC), itiles = cdiv_(M, OM);
    const int jtiles = cdiv_(N, ON2_MAX / 2);
    const int tr = cdiv_(cdiv_(N, jtiles), 8) * 8, N2 = 2 * tr;  // columns of C per tile, balanced
    const size_t bstage = (size_t)NS * N2 * 32;
    dbuf* keep = table == 1 ? &W.table_g : table == 2 ? &W.table_n : nullptr;
    dbuf* keepm = table == 1 ? &W.max_g : &W.max_n;
    bool* have = table == 1 ? &W.have_g : &W.have_n;
    const size_t abytes = (size_t)itiles * nkb * OA_STAGE;
    if (keep && !*have && (W.no_image || !image_fits(abytes) || !keepm->try_ensure((size_t)M * sizeof(unsigned long long)) ||
                           !keep->try_ensure(abytes))) {
        W.no_image = true;
        keep = nullptr;
    }
    // an operand is scaled and formatted in one launch (all of K at once) while that leaves a block
    // at most 16,384 elements (8 rows along k, 32 rows contiguous in memory) or there are blocks for
    // every SM; else maxima first, and by chunks of k.  (64 rows of 5,514 in eight blocks took 100 us
    // longer than three launches.)
    const bool onea = a.sk == 1 ? K <= 2048 || (K <= 8192 && M >= 8 * 152) : K <= 512 || M >= 32 * 152;
    const bool oneb = b.sk == 1 ? K <= 2048 || (K <= 8192 && N >= 8 * 152) : K <= 512 || N >= 32 * 152;
    // stages per chunk and row tiles per chunk of the per-call images (at most `limit` bytes each)
    int kch = nkb, ich = itiles, ztot = 0;
    auto per_split = [&](int nk) {  // stages per split of a chunk over the grid's z: fill the SMs, whole chains
        const int want = std::max(1, (N2 <= 16 ? 2 : 1) * 152 / (jtiles * std::min(ich, itiles)));
        const int splits = std::max(1, std::min({want, nk / (2 * OCHAIN), 4096}));
        return cdiv_(cdiv_(nk, splits), OCHAIN) * OCHAIN;
    };
    auto plan = [&](size_t limit) {
        kch = nkb;
        ich = itiles;
        if (!keep) {
            // long rows (Gram form): chunks of k; many rows (apply form): chunks of rows
            if ((size_t)nkb * OA_STAGE * std::min(itiles, 16) > limit)
                kch = (int)std::max<size_t>(64, limit / ((size_t)OA_STAGE * itiles));
            else
                ich = (int)std::max<size_t>(1, std::min<size_t>(itiles, limit / ((size_t)nkb * OA_STAGE)));
        }
        kch = (int)std::max<size_t>(64, std::min<size_t>(kch, limit / (bstage * jtiles)));
        kch = std::min(nkb, cdiv_(kch, OCHAIN) * OCHAIN);
        if (kch < nkb) ich = itiles;
        ztot = 0;
        for (int k0 = 0; k0 < nkb; k0 += kch) {
            const int nk = std::min(kch, nkb - k0);
            ztot += cdiv_(nk, per_split(nk));
        }
        return W.mb.try_ensure((size_t)N * sizeof(unsigned long long)) &&
               (keep || (W.ma.try_ensure((size_t)M * sizeof(unsigned long long)) &&
                         W.aimg.try_ensure((size_t)ich * kch * OA_STAGE))) &&
               W.bimg.try_ensure((size_t)jtiles * kch * bstage) &&
               (ztot == 1 || W.part.try_ensure((size_t)ztot * M * N * sizeof(double2)));
    };
    bool fits = false;
    for (size_t limit = 1ull << 30; !fits && limit >= 1ull << 24;) {
        fits = plan(limit);
        if (keep && !keep->p)  // given back for one of the buffers
            keep = nullptr, fits = false;
        else if (!fits)
            limit >>= 3;
    }
    if (!fits) return false;
    const bool whole = kch == nkb;
    unsigned long long* ma = W.ma.as<unsigned long long>();
    unsigned long long* mb = W.mb.as<unsigned long long>();
    if (keep) {
        ma = keepm->as<unsigned long long>();
        if (!*have) {
            if (onea) {
                maxfmt<false>(c, a, 0, M, K, itiles * OM, 0, nkb, 0, 0, ma, keep->as<unsigned char>());
            } else {
                row_max(c, a, M, K, ma);
                fmt<false>(c, a, 0, M, K, itiles * OM, 0, 0, nkb, 0, 0, ma, keep->as<unsigned char>());
            }
            FS_CUDA(cudaGetLastError());
            *have = true;
        }
    } else if (!(onea && whole)) {
        row_max(c, a, M, K, ma);
    }
    if (!(oneb && whole)) row_max(c, b, N, K, mb);
    OzOut o{Cd.C, Cd.cm, Cd.cn, Cd.mmap, Cd.nmap, alpha, beta, ztot > 1 ? W.part.as<double2>() : nullptr};
    const size_t sbytes = OA_STAGE + bstage;
    const auto kernel = N2 <= 16 ? oz_gemm_kernel<1> : N2 <= 32 ? oz_gemm_kernel<2> : oz_gemm_kernel<4>;
    const int nst = (int)std::min<size_t>(O_STAGES_MAX, ((N2 <= 16 ? 112 * 1024 : O_SMEM_MAX) - O_CTL) / sbytes);
    int z0 = 0;
    for (int k0 = 0; k0 < nkb; k0 += kch) {
        const int nk = std::min(kch, nkb - k0), per = per_split(nk), nz = cdiv_(nk, per);
        if (oneb && whole)
            maxfmt<true>(c, b, 0, N, K, jtiles * tr, tr, nkb, conja, conjb, mb, W.bimg.as<unsigned char>());
        else
            fmt<true>(c, b, 0, N, K, jtiles * tr, tr, k0, nk, conja, conjb, mb, W.bimg.as<unsigned char>());
        for (int i0 = 0; i0 < itiles; i0 += ich) {
            const int ni = std::min(ich, itiles - i0);
            const unsigned char* Af;
            long stride, akb;
            if (keep) {
                Af = keep->as<unsigned char>() + (size_t)i0 * nkb * OA_STAGE;
                stride = nkb;
                akb = k0;
            } else {
                if (onea && whole)
                    maxfmt<false>(c, a, i0 * OM, M, K, ni * OM, 0, nkb, 0, 0, ma, W.aimg.as<unsigned char>());
                else
                    fmt<false>(c, a, i0 * OM, M, K, ni * OM, 0, k0, nk, 0, 0, ma, W.aimg.as<unsigned char>());
                Af = W.aimg.as<unsigned char>();
                stride = nk;
                akb = 0;
            }
            for (int y0 = 0; y0 < ni; y0 += 65535) {
                const int ny = std::min(65535, ni - y0);
                kernel<<<dim3(jtiles, ny, nz), O_THREADS, (size_t)nst * sbytes + O_CTL, c->stream>>>(
                    M, N, (i0 + y0) * OM, N2, nk, per, nst, Af + (size_t)y0 * stride * OA_STAGE, stride, akb,
                    W.bimg.as<unsigned char>(), ma, mb, o, z0, ctx_errflag(c));
            }
            FS_CUDA(cudaGetLastError());
        }
        z0 += nz;
    }
    if (ztot > 1)
        oz_sum_kernel<<<cdiv_((long)M * N, 32), 256, 0, c->stream>>>(M, N, ztot, o);
    FS_CUDA(cudaGetLastError());
    return true;
}
