// Complex GEMMs of the FP32 stage on the 5th-generation tensor cores.
//
// tcgen05.mma kind::f16 with FP32 accumulators in tensor memory.  Every operand row gets a
// power of two that brings its largest component to [2^14, 2^15); a scaled component x is
// split into x_hi = fp16(x) and x_lo = fp16(x - x_hi) and the product a.b taken as
// a_hi.b_hi + a_hi.b_lo + a_lo.b_hi (three MMAs), which keeps about 22 bits of the FP32
// product (the split method of Ootomo and Yokota, 2022; components below 2^-18 of their row's
// largest are kept to 2^-40 of it).  The same products on TF32 operands (11 bits, FP32's
// exponent range, no row scale) take twice the MMA time and twice the bytes: the nonlocal
// term of 272 bands (193,673 plane waves, 2,048 projectors) 10.2 -> 5.2 ms, the error of an H
// application against 64 bits 1.0e-7 -> 0.7e-7.  What bounds it: operand stages from L2 (70
// bytes a clock and SM at 96 columns a tile).
//
// Complex arithmetic is carried by real GEMMs on interleaved (re, im) data, for
//   Gram form  C(i,j) = sum_k conj(a_ik) b_jk        (rows a_i and b_j over the long index k)
//   apply form C[i][g] = sum_k A(i,k) B[k][g]        (rows g and i over k)
// alike: UMMA A = rows m as 2K reals (re, im); UMMA B = two rows per n, so that D[m][2n] and
// D[m][2n + 1] are the real and imaginary part.  For conj(a) b these rows are (re, im) and
// (im, -re) pairs of b, for a b (re, -im) and (im, re).  The long side (plane waves, table
// rows) is always the single one, 8 bytes per complex element in the image.
//
// Formatting kernels first write each operand to global memory as the exact shared-memory
// images the MMAs read (hi and lo splits, K-major no-swizzle core-matrix layout, 16 complex k
// per stage); the projector table is formatted once per context.  The GEMM kernel then only
// moves bytes: it is persistent (one block per SM walks the (row tile, column tile, split)
// list); warp 0 issues bulk asynchronous copies (cp.async.bulk) into a ring of stages, warp 1
// issues the MMAs, and eight warps drain two accumulator buffers, so a tile's epilogue
// overlaps the next tile's copies and MMAs.
// Every mbarrier wait is bounded; on expiry the kernel raises the context's
// error flag, waits (bounded) for its copies and MMAs in flight, releases
// tensor memory and returns.
//
// The accumulation inside tensor memory loses accuracy with the length of the chain
// (measured: the error of an H application grows about linearly with it).  Every 128
// complex k the partial tile is read out and added to FP32 registers with ordinary
// round-to-nearest adds, and the next MMA starts a fresh chain.
#include "fs_beta.cuh"
#include "fs_common.cuh"

#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

namespace {

constexpr int TM = 128;                  // UMMA M (rows of the accumulator = TMEM lanes)
constexpr int TN2_MAX = 256;             // UMMA N maximum: two real rows per column of C
constexpr int KC = 16;                   // complex k per stage: 64 bytes per row and split
constexpr int A_SPLIT = TM * 64;         // one split of an A stage (8 KB)
constexpr int A_STAGE = 2 * A_SPLIT;
constexpr int CHAIN = 8;                 // stages per tensor-memory chain
constexpr int TC_THREADS = 320;
constexpr int TC_SMEM_MAX = 232448;      // the opt-in shared memory of one block
constexpr int TC_CTL = 256;              // barriers and the tensor-memory slot
constexpr int STAGES_MAX = 8;
constexpr long long WAIT_LIMIT = 1ll << 28;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// kind::f16, FP16 A and B, FP32 D, K-major both
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// bounded wait on a phase parity; returns false on timeout
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    uint32_t a = smem_u32(bar);
    for (long long it = 0; it < WAIT_LIMIT; ++it) {
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

__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem), "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void mbar_init_n(uint64_t* bar, int n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(n));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// bulk copy global -> shared (16-byte aligned, size a multiple of 16), completion on bar
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// byte offset of the 16-byte chunk (row, chunk of 4 complex k) of one split of a stage: four
// core matrices (8 rows x 16 bytes) along K per 8-row group
__host__ __device__ __forceinline__ uint32_t kmaj(int row, int chunk) {
    return (uint32_t)((((row >> 3) * 4 + chunk) << 7) + ((row & 7) << 4));
}

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)(128 >> 4) << 16;  // leading byte offset: next core matrix along K
    d |= (uint64_t)(512 >> 4) << 32;  // stride byte offset: next 8-row group
    d |= (uint64_t)1 << 46;
    return d;
}

// ---------------------------------------------------------------- operands
// element (r, k) of a GEMM operand: strided with optional row and k maps, or formed from the
// generated projectors (rows = projectors or rows = plane waves).  load4: elements k .. k + 3 of
// row r, zeros beyond R and K; called by whole warps whose lanes 4 i .. 4 i + 3 hold consecutive
// rows (a multiple of 4 first) of one chunk when rows are walked along k
template <class Op>
__device__ __forceinline__ void load4_each(const Op& op, int r, int R, int k, int K, float2 (&v)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        v[q] = make_float2(0.f, 0.f);
        if (r < R && k + q < K) v[q] = op.at(r, k + q);
    }
}
struct LdF2 {
    const float2* X;
    long sr, sk;
    const int *map, *kmap;
    const float2* const* rp = nullptr;  // rows, or k, by pointers
    const float2* const* kp = nullptr;
    __device__ __forceinline__ float2 at(int r, int k) const {
        if (rp) return rp[r][k];
        if (kp) return kp[k][r];
        return X[(map ? (long)map[r] : (long)r) * sr + (kmap ? (long)kmap[k] : (long)k) * sk];
    }
    __device__ __forceinline__ float mag(int r, int k) const {
        const float2 v = at(r, k);
        return fmaxf_nan(fabsf(v.x), fabsf(v.y));
    }
    __device__ __forceinline__ void load4(int r, int R, int k, int K, float2 (&v)[4]) const {
        load4_each(*this, r, R, k, K, v);
    }
    __device__ static __forceinline__ float fmaxf_nan(float a, float b) {  // NaN wins
        return __uint_as_float(max(__float_as_uint(a), __float_as_uint(b)));
    }
};
struct LdD2 {
    const double2* X;
    long sr, sk;
    __device__ __forceinline__ float2 at(int r, int k) const {
        const double2 v = X[(long)r * sr + (long)k * sk];
        return make_float2((float)v.x, (float)v.y);
    }
    __device__ __forceinline__ float mag(int r, int k) const {
        const float2 v = at(r, k);
        return LdF2::fmaxf_nan(fabsf(v.x), fabsf(v.y));
    }
    __device__ __forceinline__ void load4(int r, int R, int k, int K, float2 (&v)[4]) const {
        load4_each(*this, r, R, k, K, v);
    }
};
// phase e^{-i q_g.R_a} of atom a at plane wave g
__device__ __forceinline__ float2 gen_phase(const BetaGen& B, int a, int g) {
    const int code = B.gidx[g];
    const float2* ph = B.ph32 + (long)a * 3 * B.span;
    return cmul(cmul(ph[code & 1023], ph[B.span + ((code >> 10) & 1023)]), ph[2 * B.span + ((code >> 20) & 1023)]);
}
// radial factor times phase (times -i for a p type)
__device__ __forceinline__ float2 gen_value(float r, float2 e, bool p) {
    return p ? make_float2(r * e.y, -r * e.x) : make_float2(r * e.x, r * e.y);
}
struct LdGenP {  // rows: projectors
    BetaGen B;
    // the projectors of an atom share its phases: with a multiple of 4 per atom, four lanes on
    // four projectors of one atom form one phase each and exchange them (the phases were three
    // quarters of the arithmetic: H application of 96 bands of the long wire 136 -> 91 ms)
    __device__ __forceinline__ void load4(int r, int R, int k, int K, float2 (&v)[4]) const {
        if (B.nproj & 3) {
            load4_each(*this, r, R, k, K, v);
            return;
        }
        const int lane = threadIdx.x & 31, rr = min(r, R - 1), a = rr / B.nproj, c = rr - a * B.nproj;
        const float2 mine = gen_phase(B, a, min(k + (lane & 3), K - 1));
        const bool p = B.pl[c] != 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int src = (lane & ~3) | q;
            const float2 e = make_float2(__shfl_sync(0xffffffffu, mine.x, src), __shfl_sync(0xffffffffu, mine.y, src));
            v[q] = make_float2(0.f, 0.f);
            if (r < R && k + q < K) v[q] = gen_value(B.rad32[(long)c * B.npw + k + q], e, p);
        }
    }
    __device__ __forceinline__ float2 at(int r, int k) const { return beta_value32(B, r, k); }
    // (the phase has modulus one up to rounding)
    __device__ __forceinline__ float mag(int r, int k) const {
        return 1.0001f * fabsf(B.rad32[(long)(r % B.nproj) * B.npw + k]);
    }
};
struct LdGenG {  // rows: plane waves
    BetaGen B;
    // four projectors of one atom: one phase
    __device__ __forceinline__ void load4(int r, int R, int k, int K, float2 (&v)[4]) const {
        if (B.nproj & 3) {
            load4_each(*this, r, R, k, K, v);
            return;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = make_float2(0.f, 0.f);
        if (r >= R || k >= K) return;
        const int a = k / B.nproj, c = k - a * B.nproj;
        const float2 e = gen_phase(B, a, r);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = gen_value(B.rad32[(long)(c + q) * B.npw + r], e, B.pl[c + q] != 0);
    }
    __device__ __forceinline__ float2 at(int r, int k) const { return beta_value32(B, k, r); }
    __device__ __forceinline__ float mag(int r, int k) const {
        return 1.0001f * fabsf(B.rad32[(long)(k % B.nproj) * B.npw + r]);
    }
};

// scale 2^s of a row from its largest magnitude: 2^(15 - E) with |x| < 2^E, as a float
__device__ __forceinline__ float row_scale(uint32_t bits) {
    const int e = (int)(bits >> 23) - 126;
    const int s = max(-126, min(126, 15 - e));
    return __uint_as_float((uint32_t)(s + 127) << 23);
}
__device__ __forceinline__ float row_unscale(uint32_t bits) {
    const int e = (int)(bits >> 23) - 126;
    const int s = max(-126, min(126, 15 - e));
    return __uint_as_float((uint32_t)(127 - s) << 23);
}

// largest magnitude (as bits) of every row over k in [0, K); kcont: a warp walks along k, else a
// thread per row
template <class Op>
__global__ void tc_max_kernel(Op op, int R, int K, int kper, int kcont, uint32_t* __restrict__ out) {
    const int k0 = blockIdx.y * kper, k1 = min(K, k0 + kper);
    if (kcont) {
        const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (r >= R) return;
        uint32_t m = 0;
#pragma unroll 4
        for (int k = k0 + lane; k < k1; k += 32) m = max(m, __float_as_uint(op.mag(r, k)));
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) atomicMax(out + r, m);
    } else {
        const int r = blockIdx.x * blockDim.x + threadIdx.x;
        if (r >= R) return;
        uint32_t m = 0;
#pragma unroll 4
        for (int k = k0; k < k1; ++k) m = max(m, __float_as_uint(op.mag(r, k)));
        atomicMax(out + r, m);
    }
}

// The 16-byte chunk ch (4 complex k) of local row lr (operand row r) in both splits.
//   BSIDE = false: A image, tiles of 128 rows
//   BSIDE = true : B image, tiles of tr operand rows, two image rows each; conja: conj(a) b
template <bool BSIDE, class Op>
__device__ __forceinline__ void put_chunk(const Op& op, int lr, int r, int R, int ch, int K, int tr, int kb0, int nkb,
                                          int conja, float s, unsigned char* __restrict__ out) {
    const uint32_t split = BSIDE ? (uint32_t)tr * 128 : (uint32_t)A_SPLIT;
    const int k = kb0 * KC + 4 * ch;
    float2 v[4];
    op.load4(r, R, k, K, v);
    uint32_t h[4], l[4];  // (re, im) pairs of the hi and lo parts
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float x = v[q].x * s, y = v[q].y * s;
        const __half2 hh = __floats2half2_rn(x, y);
        const float2 hf = __half22float2(hh);
        const __half2 ll = __floats2half2_rn(x - hf.x, y - hf.y);
        h[q] = *reinterpret_cast<const uint32_t*>(&hh);
        l[q] = *reinterpret_cast<const uint32_t*>(&ll);
    }
    const int kb = ch >> 2, cc = ch & 3;
    if (!BSIDE) {
        unsigned char* st = out + ((long)(lr / TM) * nkb + kb) * A_STAGE + kmaj(lr % TM, cc);
        *reinterpret_cast<uint4*>(st) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(st + A_SPLIT) = make_uint4(l[0], l[1], l[2], l[3]);
    } else {
        const int tile = lr / tr, j = lr - tile * tr;
        unsigned char* st = out + ((long)tile * nkb + kb) * (2l * split) + kmaj(2 * j, cc);
        const uint32_t s0 = conja ? 0u : 0x80000000u, s1 = conja ? 0x80000000u : 0u;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            uint32_t a[4], b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t p = u ? l[q] : h[q];
                a[q] = p ^ s0;                          // (re, im) or (re, -im)
                b[q] = __byte_perm(p, p, 0x1032) ^ s1;  // (im, -re) or (im, re)
            }
            *reinterpret_cast<uint4*>(st + u * split) = make_uint4(a[0], a[1], a[2], a[3]);
            *reinterpret_cast<uint4*>(st + u * split + 16) = make_uint4(b[0], b[1], b[2], b[3]);
        }
    }
}

// Images of rows r0 .., stages [kb0, kb0 + nkb) as local stages 0 .. nkb, by known maxima
template <bool BSIDE, class Op>
__global__ void tc_fmt_kernel(Op op, int kcont, int r0, int R, int K, int rows, int tr, int kb0, int nkb, int conja,
                              const uint32_t* __restrict__ rmax, unsigned char* __restrict__ out) {
    const long nch = 4l * nkb, total = (long)rows * nch;  // rows is a multiple of 8
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        int lr, ch;
        if (kcont) {  // 8 rows x 4 chunks (one stage) per warp
            const int lane = (int)(t & 31);
            const long w = t >> 5;
            lr = (int)(w / nkb) * 8 + (lane & 7);
            ch = (int)(w % nkb) * 4 + (lane >> 3);
        } else {
            lr = (int)(t % rows);
            ch = (int)(t / rows);
        }
        const int r = r0 + lr;
        put_chunk<BSIDE>(op, lr, r, R, ch, K, tr, kb0, nkb, conja, r < R ? row_scale(rmax[r]) : 0.f, out);
    }
}

// Short rows: maxima and images of 8 rows per block in one launch (a warp finds a row's maximum)
template <bool BSIDE, class Op>
__global__ void __launch_bounds__(256) tc_maxfmt_kernel(Op op, int R, int K, int tr, int nkb, int conja,
                                                        uint32_t* __restrict__ rmax, unsigned char* __restrict__ out) {
    __shared__ float scale[8];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, lr0 = blockIdx.x * 8;
    uint32_t m = 0;
    if (lr0 + w < R)
#pragma unroll 4
        for (int k = lane; k < K; k += 32) m = max(m, __float_as_uint(op.mag(lr0 + w, k)));
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
        scale[w] = row_scale(m);
        if (lr0 + w < R) rmax[lr0 + w] = m;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 32 * nkb; t += 256) {
        const int lr = lr0 + (t & 7);
        put_chunk<BSIDE>(op, lr, lr, R, t >> 3, K, tr, 0, nkb, conja, scale[t & 7], out);
    }
}

// Rows contiguous in memory (k strided): maxima (over kmax of the k) and images of 32 rows per
// block in one launch; a warp takes every eighth k (then every eighth chunk) of all 32 rows, and
// the second reading comes from L1
template <bool BSIDE, class Op>
__global__ void __launch_bounds__(256) tc_maxfmt_rows_kernel(Op op, int r0, int R, int K, int kmax, int rows, int tr,
                                                             int nkb, int conja, uint32_t* __restrict__ rmax,
                                                             unsigned char* __restrict__ out) {
    __shared__ uint32_t part[8][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, lr = blockIdx.x * 32 + lane, r = r0 + lr;
    uint32_t m = 0;
    if (r < R)
#pragma unroll 4
        for (int k = w; k < kmax; k += 8) m = max(m, __float_as_uint(op.mag(r, k)));
    part[w][lane] = m;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) m = max(m, part[i][lane]);
    if (w == 0 && r < R) rmax[r] = m;
    const float s = row_scale(m);
    if (lr < rows)
        for (int ch = w; ch < 4 * nkb; ch += 8) put_chunk<BSIDE>(op, lr, r, R, ch, K, tr, 0, nkb, conja, s, out);
}

// ---------------------------------------------------------------- the GEMM
// Where a tile goes: partial sums part[((z0 + z) N + n) M + m] (raw, FP32), or
// C[nmap(n) ldc + m] = alpha acc + beta D[..].
struct TcOut {
    float2* part;
    float2* C;
    long ldc;
    const int* nmap;
    const float2* D;
    long ldd;
    float alpha, beta;
};

// Tile t: column tile t mod jtiles, then row tile, then split (blocks that share a row tile
// run side by side, so its image comes from L2 after the first).  Split z takes stages
// [z kbs, min(nkb, (z + 1) kbs)).
__global__ void __launch_bounds__(TC_THREADS, 1)
tc_gemm_kernel(int M, int N, int m0, int N2, int itiles, int jtiles, int ntiles, int nkb, int kbs, int nst,
               int lower, const unsigned char* __restrict__ Af, long a_stride, long a_kb0, const unsigned char* __restrict__ Bf,
               const uint32_t* __restrict__ ma, const uint32_t* __restrict__ mb, TcOut o, int z0, int* errflag) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t bsplit = (uint32_t)N2 * 64, sbytes = A_STAGE + 2 * bsplit;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)nst * sbytes);
    uint64_t* empty = full + nst;
    uint64_t* accf = empty + nst;
    uint64_t* acce = accf + 2;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(acce + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            mbar_init_n(&full[s], 1);
            mbar_init_n(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init_n(&accf[b], 1);
            mbar_init_n(&acce[b], 8);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            long long g = 0;  // stages issued by this block
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
                const int jt = tile % jtiles, it = (tile / jtiles) % itiles, kb0 = tile / (jtiles * itiles) * kbs;
                if (lower && jt * (N2 >> 1) >= (it + 1) * TM) continue;  // wholly above the diagonal
                const int nk = min(nkb, kb0 + kbs) - kb0;
                const unsigned char* a = Af + ((long)it * a_stride + a_kb0 + kb0) * A_STAGE;
                const unsigned char* b = Bf + ((long)jt * nkb + kb0) * (2l * bsplit);
                for (int kb = 0; kb < nk; ++kb, ++g) {
                    const int st = (int)(g % nst);
                    if (g >= nst && !mbar_wait(&empty[st], (uint32_t)((g / nst) - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    unsigned char* dst = smem + (size_t)st * sbytes;
                    mbar_expect_tx(&full[st], sbytes);
                    bulk_g2s(dst, a + (long)kb * A_STAGE, A_STAGE, &full[st]);
                    bulk_g2s(dst + A_STAGE, b + (long)kb * (2l * bsplit), 2 * bsplit, &full[st]);
                }
            }
            // every copy issued has landed before the block can exit
            for (long long q = g > nst ? g - nst : 0; q < g; ++q)
                if (!mbar_wait(&full[q % nst], (uint32_t)(q / nst) & 1)) ok = false;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_f16(TM, N2);
            long long g = 0, last = -1;
            int ch = 0;  // accumulator chains started by this block
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
                const int jt = tile % jtiles, it = (tile / jtiles) % itiles;
                if (lower && jt * (N2 >> 1) >= (it + 1) * TM) continue;
                const int kb0 = tile / (jtiles * itiles) * kbs, nk = min(nkb, kb0 + kbs) - kb0;
                for (int kb = 0; kb < nk; ++kb, ++g) {
                    const int st = (int)(g % nst), buf = ch & 1;
                    const bool first = kb % CHAIN == 0;
                    if (!mbar_wait(&full[st], (uint32_t)(g / nst) & 1)) {
                        ok = false;
                        break;
                    }
                    if (first && ch >= 2 && !mbar_wait(&acce[buf], ((ch >> 1) - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t base = smem_u32(smem + (size_t)st * sbytes);
                    const uint64_t ahi = sdesc(base), alo = ahi + (A_SPLIT >> 4);
                    const uint64_t bhi = sdesc(base + A_STAGE), blo = bhi + (bsplit >> 4);
                    const uint32_t d = tmem + (uint32_t)(buf * 256);
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks) {  // 16 reals each: two core matrices
                        const uint64_t w = (uint64_t)(ks * 256) >> 4;
                        mma_f16(d, ahi + w, bhi + w, idesc, (first && ks == 0) ? 0u : 1u);
                        mma_f16(d, ahi + w, blo + w, idesc, 1u);
                        mma_f16(d, alo + w, bhi + w, idesc, 1u);
                    }
                    mma_commit(&empty[st]);
                    if (kb % CHAIN == CHAIN - 1 || kb == nk - 1) {
                        mma_commit(&accf[buf]);
                        ++ch;
                    }
                    last = g;
                }
            }
            // the MMAs issued have completed before tensor memory is released
            if (last >= 0 && !mbar_wait(&empty[last % nst], (uint32_t)(last / nst) & 1)) ok = false;
        }
    } else {
        // thread: TMEM lane 32 (warp & 3) + lane, accumulator columns 128 h + 32 j + e
        const int q = warp & 3, h = (warp - 2) >> 2;
        int ch = 0;
        float acc[4][32];
        for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
            const int jt = tile % jtiles, it = (tile / jtiles) % itiles, z = tile / (jtiles * itiles);
            if (lower && jt * (N2 >> 1) >= (it + 1) * TM) continue;
            const int nk = min(nkb, (z + 1) * kbs) - z * kbs, nchain = (nk + CHAIN - 1) / CHAIN;
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[j][e] = 0.f;
            for (int cc = 0; cc < nchain; ++cc, ++ch) {
                const int buf = ch & 1;
                // every lane polls; the vote keeps the warp together if one gives up
                if (!__all_sync(0xffffffffu, mbar_wait(&accf[buf], (ch >> 1) & 1))) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c0 = 128 * h + 32 * j;
                    if (c0 < N2) {  // warp-uniform
                        float v[32];
                        tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * 256 + c0), v);
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[j][e] += v[e];
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&acce[buf]);
            }
            if (!ok) break;
            const int m = m0 + it * TM + 32 * q + lane;
            if (m >= M) continue;
            const float fa = row_unscale(ma[m]);
            const int n0 = jt * (N2 >> 1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int nb = n0 + 64 * h + 16 * j;              // first column of C of this group
                const int nn = min(16, min(n0 + (N2 >> 1), N) - nb);
                if (nn <= 0) continue;  // warp-uniform
                if (o.part) {
                    float2* out = o.part + ((long)(z0 + z) * N + nb) * M + m;
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (e < nn) {
                            const float fb = row_unscale(mb[nb + e]);
                            out[(long)e * M] = make_float2(acc[j][2 * e] * fa * fb, acc[j][2 * e + 1] * fa * fb);
                        }
                } else {
                    // in groups of 8 outputs: the row indices, then the D values, then the stores,
                    // so that the loads of a group are in flight together (D may be C itself;
                    // each thread reads only the elements it writes)
#pragma unroll
                    for (int e0 = 0; e0 < 16; e0 += 8) {
                        long row[8];
                        float2 dv[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const int n = nb + e0 + e;
                            row[e] = e0 + e < nn ? (o.nmap ? (long)__ldg(o.nmap + n) : (long)n) : -1;
                        }
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            dv[e] = make_float2(0.f, 0.f);
                            if (o.beta != 0.f && row[e] >= 0) dv[e] = o.D[row[e] * o.ldd + m];
                        }
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            if (row[e] >= 0) {
                                const float fb = row_unscale(mb[nb + e0 + e]);
                                float x = o.alpha * (acc[j][2 * (e0 + e)] * fa * fb);
                                float y = o.alpha * (acc[j][2 * (e0 + e) + 1] * fa * fb);
                                if (o.beta != 0.f) {
                                    x += o.beta * dv[e].x;
                                    y += o.beta * dv[e].y;
                                }
                                o.C[row[e] * o.ldc + m] = make_float2(x, y);
                            }
                    }
                }
            }
        }
    }
    if (!ok) *(volatile int*)errflag = 1;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// C(m, n) = alpha sum_z part(z, n, m) + beta C(m, n) in FP64: 32 outputs per block, eight groups of
// consecutive z added in order (deterministic); lower: outputs of
// skipped tiles (tr columns wide) stay as they are
__global__ void __launch_bounds__(256) tc_sum_kernel(int M, int N, int splits, const float2* __restrict__ part,
                                                     double2* C, long cm, long cn, double alpha, double beta,
                                                     int lower, int tr) {
    __shared__ double2 sh[8][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long total = (long)M * N, t = blockIdx.x * 32l + lane;
    const long n = t / M, m = t - n * M;
    const bool live = t < total && !(lower && n / tr * tr >= (m / TM + 1) * TM);
    const int per = (splits + 7) / 8, z1 = min(splits, (w + 1) * per);
    double sx = 0, sy = 0;
    if (live)
#pragma unroll 8
        for (int z = w * per; z < z1; ++z) {
            const float2 v = part[(long)z * total + t];
            sx += v.x;
            sy += v.y;
        }
    sh[w][lane] = make_double2(sx, sy);
    __syncthreads();
    if (w || !live) return;
    double2 s = sh[0][lane];
    for (int i = 1; i < 8; ++i) s = cadd(s, sh[i][lane]);
    double2* dst = C + m * cm + n * cn;
    double2 o = make_double2(alpha * s.x, alpha * s.y);
    if (beta != 0.0) {
        o.x += beta * dst->x;
        o.y += beta * dst->y;
    }
    *dst = o;
}

// The bounded wait of the pipelines, on a barrier that nothing completes: it
// polls `limit` times, gives up and raises the context's error flag.
__global__ void wait_selftest_kernel(long long limit, int* errflag) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init_n(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t a = smem_u32(&bar);
        bool ok = false;
        for (long long it = 0; it < limit && !ok; ++it) {
            uint32_t r;
            asm volatile(
                "{\n\t.reg .pred p;\n\t"
                "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}"
                : "=r"(r)
                : "r"(a), "r"(0u)
                : "memory");
            ok = r != 0;
        }
        if (!ok) *(volatile int*)errflag = 1;
    }
}

inline int cdiv_(long a, long b) { return (int)((a + b - 1) / b); }

// row maxima over k in [0, K)
template <class Op> void tc_row_max(fs_ctx* c, const Op& op, int kcont, int R, int K, uint32_t* out) {
    FS_CUDA(cudaMemsetAsync(out, 0, (size_t)R * sizeof(uint32_t), c->stream));
    const int bx = kcont ? cdiv_(R, 8) : cdiv_(R, 256);
    const int by = std::min(65535, std::max(1, std::min(cdiv_(K, 128), 152 * 16 / std::max(1, bx))));
    tc_max_kernel<Op><<<dim3(bx, by), 256, 0, c->stream>>>(op, R, K, cdiv_(K, by), kcont, out);
}

// maxima of the first `have` rows repeated over the others
__global__ void tc_repeat_kernel(uint32_t* m, int have, int R) {
    const int r = have + blockIdx.x * blockDim.x + threadIdx.x;
    if (r < R) m[r] = m[r % have];
}
// projectors of one type have the same radial factor: nproj rows stand for all
void tc_row_max(fs_ctx* c, const LdGenP& op, int kcont, int R, int K, uint32_t* out) {
    const int have = std::min(R, op.B.nproj);
    tc_row_max<LdGenP>(c, op, kcont, have, K, out);
    if (R > have) tc_repeat_kernel<<<cdiv_(R - have, 256), 256, 0, c->stream>>>(out, have, R);
}

template <bool BSIDE, class Op>
void tc_fmt(fs_ctx* c, const Op& op, int kcont, int r0, int R, int K, int rows, int tr, int kb0, int nkb, int conja,
            const uint32_t* rmax, unsigned char* out) {
    const long thr = (long)rows * 4 * nkb;
    tc_fmt_kernel<BSIDE, Op><<<(int)std::min<long>(152 * 16, (thr + 255) / 256), 256, 0, c->stream>>>(
        op, kcont, r0, R, K, rows, tr, kb0, nkb, conja, rmax, out);
}

// The GEMM over operand a (rows m, 128 a tile; image kept in `keep` with its maxima in `keepm`
// when given) and b (rows n); acont / bcont: contiguous along k (both in the Gram form), amaxk: k
// over which a's row maxima are taken (a generated table repeats its first nproj types).
// d64: FP64 result through split-K partial sums; else the FP32 result goes where o says.
struct TcDst64 {
    double2* C;
    long cm, cn;
    double alpha, beta;
};
template <class OpA, class OpB>
void tc_run(fs_ctx* c, int M, int N, int K, const OpA& a, int acont, int amaxk, const OpB& b, int bcont, int conja,
            dbuf* keep, dbuf* keepm, const TcDst64* d64, TcOut o, int lower = 0) {
    smem_limit(c->tc_limit, TC_SMEM_MAX, {(const void*)tc_gemm_kernel});
    const int nkb = std::max(1, cdiv_(K, KC)), itiles = cdiv_(M, TM);
    const int jtiles = cdiv_(N, TN2_MAX / 2);
    const int tr = cdiv_(cdiv_(N, jtiles), 8) * 8, N2 = 2 * tr;  // columns of C per tile, balanced
    const size_t bstage = (size_t)2 * N2 * 64;
    if (keep && !keep->p && (size_t)itiles * nkb * A_STAGE > FS_TABLE_FMT_MAX_BYTES) keep = nullptr;
    c->tc_ma.ensure((size_t)M * sizeof(uint32_t));
    c->tc_mb.ensure((size_t)N * sizeof(uint32_t));
    uint32_t *ma = c->tc_ma.as<uint32_t>(), *mb = c->tc_mb.as<uint32_t>();
    // How an operand is scaled and formatted: rows contiguous in memory, in one launch; short rows
    // along k (up to 4,096: a block's two passes over 8 rows take less than three launches), in
    // one launch; long rows along k, maxima first, so that the images can be made by chunks of k
    const bool shortk = K <= 4096 && (size_t)nkb * (itiles * A_STAGE + jtiles * bstage) <= FS_FMT_CHUNK_BYTES;
    const bool onea = !acont || shortk, oneb = !bcont || shortk;
    auto format_a = [&](int i0, int ni, int k0, int nk, uint32_t* mx, unsigned char* dst) {
        if (!acont)
            tc_maxfmt_rows_kernel<false, OpA><<<ni * TM / 32, 256, 0, c->stream>>>(a, i0 * TM, M, K, amaxk, ni * TM, 0,
                                                                                  nkb, 0, mx, dst);
        else if (onea)
            tc_maxfmt_kernel<false, OpA><<<ni * TM / 8, 256, 0, c->stream>>>(a, M, K, 0, nkb, 0, mx, dst);
        else
            tc_fmt<false>(c, a, acont, i0 * TM, M, K, ni * TM, 0, k0, nk, 0, mx, dst);
    };
    if (keep) {
        if (!keep->p) {
            keepm->ensure((size_t)M * sizeof(uint32_t));
            keep->alloc((size_t)itiles * nkb * A_STAGE);
            if (!onea) tc_row_max(c, a, acont, M, amaxk, keepm->as<uint32_t>());
            format_a(0, itiles, 0, nkb, keepm->as<uint32_t>(), keep->as<unsigned char>());
        }
        ma = keepm->as<uint32_t>();
    } else if (!onea) {
        tc_row_max(c, a, acont, M, amaxk, ma);
    }
    if constexpr (std::is_same_v<OpA, LdF2> && std::is_same_v<OpB, LdF2>) {
        // the Gram matrix of one set of rows: one set of maxima
        if (!oneb && !onea && !keep && a.rp && a.rp == b.rp && M == N) mb = ma;
    }
    if (!oneb && mb != ma) tc_row_max(c, b, bcont, N, K, mb);
    // per-call images in chunks of at most FS_FMT_CHUNK_BYTES: along k for a split result, along
    // the rows of a otherwise
    int kch = nkb, ich = itiles;
    if (d64 && !shortk)
        kch = (int)std::max<size_t>(16, std::min<size_t>(nkb, FS_FMT_CHUNK_BYTES / ((keep ? 0 : (size_t)itiles * A_STAGE) +
                                                                                   jtiles * bstage)));
    else if (!d64 && !keep)
        ich = (int)std::max<size_t>(1, std::min<size_t>(itiles, FS_FMT_CHUNK_BYTES / ((size_t)nkb * A_STAGE)));
    // split of a chunk over K (at least two chains each): the fewest splits with which the tiles
    // come to whole rounds over the SMs but for 7 %, else those with the least idle time (48
    // tiles of the wire's projections: 3 splits = 144 tiles instead of 7 = 336, which left the
    // third round of blocks a fifth full)
    const int tiles = lower ? std::max(1, (itiles * jtiles + std::max(itiles, jtiles)) / 2) : itiles * jtiles;
    auto per_split = [&](int nk) {
        int best = 1;
        if (d64) {
            double eff_best = 0;
            const int most = std::max(1, std::min(nk / (2 * CHAIN), cdiv_(4 * c->nsm, tiles)));
            for (int sp = 1; sp <= most; ++sp) {
                const double eff = (double)tiles * sp / ((double)cdiv_((long)tiles * sp, c->nsm) * c->nsm);
                if (eff > eff_best + 1e-9) {
                    eff_best = eff;
                    best = sp;
                }
                if (eff >= 0.93) break;
            }
        }
        return cdiv_(nk, best);
    };
    int ztot = 0;
    if (d64) {
        for (int k0 = 0; k0 < nkb; k0 += kch) {
            const int nk = std::min(kch, nkb - k0);
            ztot += cdiv_(nk, per_split(nk));
        }
        c->splitk.ensure((size_t)ztot * M * N * sizeof(float2));
        o.part = c->splitk.as<float2>();
    }
    const size_t sbytes = A_STAGE + bstage;
    const int nst = (int)std::min<size_t>(STAGES_MAX, (TC_SMEM_MAX - TC_CTL) / sbytes);
    int z0 = 0;
    for (int k0 = 0; k0 < nkb; k0 += kch) {
        const int nk = std::min(kch, nkb - k0), per = per_split(nk), nz = cdiv_(nk, per);
        c->bfmt.ensure((size_t)jtiles * nk * bstage);
        if (!bcont)
            tc_maxfmt_rows_kernel<true, OpB><<<cdiv_((long)jtiles * tr, 32), 256, 0, c->stream>>>(
                b, 0, N, K, K, jtiles * tr, tr, nkb, conja, mb, c->bfmt.as<unsigned char>());
        else if (oneb)
            tc_maxfmt_kernel<true, OpB><<<jtiles * tr / 8, 256, 0, c->stream>>>(b, N, K, tr, nkb, conja, mb,
                                                                               c->bfmt.as<unsigned char>());
        else
            tc_fmt<true>(c, b, bcont, 0, N, K, jtiles * tr, tr, k0, nk, conja, mb, c->bfmt.as<unsigned char>());
        for (int i0 = 0; i0 < itiles; i0 += ich) {
            const int ni = std::min(ich, itiles - i0);
            const unsigned char* Af;
            long stride = nk, akb = 0;
            if (keep) {
                Af = keep->as<unsigned char>() + (size_t)i0 * nkb * A_STAGE;
                stride = nkb;
                akb = k0;
            } else {
                c->afmt.ensure((size_t)ni * nk * A_STAGE);
                format_a(i0, ni, k0, nk, ma, c->afmt.as<unsigned char>());
                Af = c->afmt.as<unsigned char>();
            }
            const int ntiles = jtiles * ni * nz, grid = std::min(ntiles, c->nsm);
            tc_gemm_kernel<<<grid, TC_THREADS, (size_t)nst * sbytes + TC_CTL, c->stream>>>(
                M, N, i0 * TM, N2, ni, jtiles, ntiles, nk, per, nst, lower, Af, stride, akb, c->bfmt.as<unsigned char>(), ma,
                mb, o, z0, ctx_errflag(c));
            FS_CUDA(cudaGetLastError());
        }
        z0 += nz;
    }
    if (d64)
        tc_sum_kernel<<<cdiv_((long)M * N, 32), 256, 0, c->stream>>>(M, N, ztot, o.part, d64->C, d64->cm, d64->cn,
                                                                     d64->alpha, d64->beta, lower, tr);
    FS_CUDA(cudaGetLastError());
}

}  // namespace

void tc_gemm_gram(fs_ctx* c, int M, int N, int K, const float2* A, long lda, const int* amap, const float2* B,
                  long ldb, const int* bmap, double2* C, long ci, long cj, double alpha, double beta, int kid,
                  const BetaGen* gen) {
    if (M <= 0 || N <= 0) return;
    ProfScope ps(c, kid, ((double)M + N) * K * sizeof(float2) + (double)M * N * sizeof(double2), 8.0 * M * N * K);
    const LdF2 b{B, ldb, 1, bmap, nullptr};
    const TcDst64 d{C, ci, cj, alpha, beta};
    if (gen) {
        tc_run(c, M, N, K, LdGenP{*gen}, 1, K, b, 1, 1, nullptr, nullptr, &d, TcOut{});
        return;
    }
    const LdF2 a{A, lda, 1, amap, nullptr};
    const bool table = A == c->beta32.as<float2>() && !amap && M == c->nptot && K == c->npw;
    tc_run(c, M, N, K, a, 1, K, b, 1, 1, table ? &c->beta32_gfmt : nullptr, &c->tc_gmax, &d, TcOut{});
}

void tc_gemm_gram_rows(fs_ctx* c, int n, int K, const float2* const* A, const float2* const* B, double2* C, int lower) {
    if (n <= 0) return;
    ProfScope ps(c, KS_GRAM, 2.0 * n * K * sizeof(float2) + (double)n * n * sizeof(double2), 8.0 * n * n * K);
    const TcDst64 d{C, 1, n, 1.0, 0.0};
    tc_run(c, n, n, K, LdF2{nullptr, 0, 1, nullptr, nullptr, A}, 1, K, LdF2{nullptr, 0, 1, nullptr, nullptr, B}, 1, 1,
           nullptr, nullptr, &d, TcOut{}, lower);
}

void tc_gemm_nn_rows(fs_ctx* c, int M, int N, int K, const double2* A, long ai, const float2* const* B, float2* C,
                     long ldc) {
    if (M <= 0 || N <= 0) return;
    ProfScope ps(c, KS_ROTATE, ((double)K + M) * N * sizeof(float2) + (double)M * K * sizeof(double2), 8.0 * M * N * K);
    tc_run(c, N, M, K, LdF2{nullptr, 1, 0, nullptr, nullptr, nullptr, B}, 0, K, LdD2{A, ai, 1}, 1, 0, nullptr, nullptr,
           nullptr, TcOut{nullptr, C, ldc, nullptr, nullptr, 0, 1.f, 0.f});
}

template <typename A2>
void tc_gemm_nn(fs_ctx* c, int M, int N, int K, const A2* A, long ai, long ak, const float2* B, long ldb,
                const int* bmap, float2* C, long ldc, const int* cmap, double alpha, double beta, const float2* D,
                long ldd, int kid, const BetaGen* gen) {
    if (M <= 0 || N <= 0) return;
    ProfScope ps(c, kid, ((double)K + M * (beta != 0.0 ? 2.0 : 1.0)) * N * sizeof(float2) + (double)M * K * sizeof(A2),
                 8.0 * M * N * K);
    const TcOut o{nullptr, C, ldc, cmap, D, ldd, (float)alpha, (float)beta};
    auto go = [&](const auto& co) {
        if (gen) {  // (every type occurs among the first nproj projectors)
            tc_run(c, N, M, K, LdGenG{*gen}, 0, std::min(K, gen->nproj), co, ak == 1, 0, nullptr, nullptr, nullptr, o);
            return;
        }
        const LdF2 b{B, 1, ldb, nullptr, bmap};
        const bool table = B == c->beta32.as<float2>() && !bmap && N == c->npw && K == c->nptot;
        tc_run(c, N, M, K, b, 0, K, co, ak == 1, 0, table ? &c->beta32_fmt : nullptr, &c->tc_nmax, nullptr, o);
    };
    if constexpr (sizeof(A2) == 16)
        go(LdD2{A, ai, ak});
    else
        go(LdF2{A, ai, ak, nullptr, nullptr});
}

template void tc_gemm_nn<double2>(fs_ctx*, int, int, int, const double2*, long, long, const float2*, long, const int*,
                                  float2*, long, const int*, double, double, const float2*, long, int, const BetaGen*);
template void tc_gemm_nn<float2>(fs_ctx*, int, int, int, const float2*, long, long, const float2*, long, const int*,
                                 float2*, long, const int*, double, double, const float2*, long, int, const BetaGen*);

namespace {
fs_status wait_selftest(fs_ctx* c, long long polls, bool pending) {
    if (!c) return FS_ERR_ARG;
    if (polls < 1 || polls > (1ll << 24)) {
        c->err = "fs_wait_selftest: polls out of range [1, 2^24]";
        return FS_ERR_ARG;
    }
    if (pending) {
        wait_selftest_kernel<<<1, 32, 0, c->stream>>>(polls, ctx_errflag(c));
        return cudaGetLastError() == cudaSuccess ? FS_OK : FS_ERR_CUDA;
    }
    return ctx_call(c, [&] {
        wait_selftest_kernel<<<1, 32, 0, c->stream>>>(polls, ctx_errflag(c));
        FS_CUDA(cudaGetLastError());
    });
}
}  // namespace

extern "C" fs_status fs_wait_selftest(fs_ctx* c, long long polls) { return wait_selftest(c, polls, false); }
extern "C" fs_status fs_wait_selftest_pending(fs_ctx* c, long long polls) { return wait_selftest(c, polls, true); }
