// FP64 complex contraction on the 5th-generation tensor cores: the operands
// are cut into 8-bit digits and the digit products, integers that an FP32
// accumulator holds exactly, run as bf16 tcgen05.mma (the Ozaki scheme:
// Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", Numer.
// Algorithms 59, 2012; on tensor cores: Mukunoki et al., ISC 2020).
//
// Numbers.  Row p of P (row q of Q) has one exponent E: |x| < 2^E over the
// row.  x = 2^(E - 55) t with |t| <= 2^55 an integer (x rounded to the row's
// grid; entries within 2^-2 of the row's largest are exact), t = sum_i d_i
// 256^(6-i), i = 0..6, d_i in [-128, 128].  A product sums the levels
//   v_l = sum_{i+j=l} sum_k d_i(p, k) d_j(q, k),  l = 0..7,
//   sum_k t t' ~ 256^5 sum_l 256^(7-l) v_l   (levels 8..12, below 2^-60 of the
//   largest product, are dropped).
// |v_l| <= 7 * 128 * 2^14 < 2^24 for 128 values of k, so the FP32
// accumulation of a K chunk of 128 reals has no rounding at all; chunks are
// added in 64-bit integers, and the one rounding of the result is the final
// conversion to FP64.
//
// Accuracy.  What is lost is the part of an entry below its row's grid:
//   |error| <= 2^-56 (2^Ep sum_k |q_k| + 2^Eq sum_k |p_k|) + K 2^-60 2^(Ep + Eq).
// For operands of one size along K that is less than the roundings of an FMA
// chain (uniform operands, rms relative to |row||column|: 7e-18 at K = 64, the
// chain 3.3e-17).  Not so where small entries of one row meet large ones of
// the other: graded against each other over 2^32, digits alone are off by
// 2e-8 of sum |p_k||q_k|.  So digit_check_kernel computes a lower bound of
// sum_k |p_k||q_k| for every output (a bf16 product of the magnitudes, a
// hundredth of the work) and marks the outputs whose error bound above exceeds
// that of an FMA chain, 2 K 2^-53 sum |p_k||q_k|; digit_fix_kernel computes
// those by FMA chains.  Every output so has an FMA chain's bound, whatever the
// operands hold.  Callers whose analysis needs no more than |row||column|
// (the panel QR, whose operands are columns of norm about 1) leave the check
// out (elementwise = false).  The check costs 7 us of a small contraction and 6
// to 11 % of a large one (4096 x 64 x 64 48 -> 55 us, 16384 x 128 x 128 180 -> 200);
// in steps and observables of this library 0 to 0.02 % of the outputs are marked.
//
// Why: GB300's FP64 pipe gives 1.06 TFLOP/s; 34 bf16 products give one FP64
// product at up to 1908 / 34 = 56 TFLOP/s.  Measured, packing and check included,
// against the FMA kernels: 16384 x 128 x 128 in batches of 16 28.1 -> 1.19 ms (28.9
// TFLOP/s), 128 x 128 x 16384 in batches of 16 from a product state 40 -> 2.75 ms
// (1.65 before the outputs were checked), 4096 x 64 x 64 in batches of 4 464 -> 58
// us, 64 x 4096 x 256 463 -> 91 us.
//
// Complex numbers use the real embedding of gemm_split.cu: P rows hold
// (Re, Im) pairs, Q rows 2n and 2n + 1 hold (Re, -Im) and (Im, Re).
//
// Kernel.  Persistent, one CTA per SM, 18 warps: warp 16 loads 32-wide K
// slices of all 7 digit planes of both sides (one 3-D TMA box each, 64-byte
// swizzle) into a 2-stage ring (84 KB per stage), warp 17 issues the 34 digit
// products, level by level, into 8 TMEM accumulators of 64 columns (all 512),
// warps 0-15 drain.  A chunk's level is released as soon as it is drained, so
// the next chunk's low levels run while the last ones are drained; the
// conversion to FP64 is integer arithmetic (the FP64 pipe would take longer
// than the MMAs) and overlaps the next tile's MMAs.
#include "common.cuh"
#include "tcgen05.cuh"

#include <algorithm>
#include <cstring>
#include <math_constants.h>

namespace {

constexpr int ND = 7;            // digits
constexpr int NLEV = 8;          // levels kept
constexpr int BM = 128, BN = 64; // tile: P rows x real Q rows
constexpr int BK = 32;           // real K per stage (64 bytes of bf16)
constexpr int STAGES = 2;
constexpr int CHUNK_ST = 4;      // stages per exact chunk (128 real K)
constexpr int P_PLANE = BM * BK * 2, Q_PLANE = BN * BK * 2;
constexpr int P_BYTES = ND * P_PLANE, STAGE_BYTES = ND * (P_PLANE + Q_PLANE);
constexpr int DRAIN_WARPS = 16, DRAIN_THREADS = 32 * DRAIN_WARPS;
constexpr int TMA_WARP = DRAIN_WARPS, MMA_WARP = DRAIN_WARPS + 1;
constexpr int THREADS = DRAIN_THREADS + 64;
constexpr int DCOLS = BN / (DRAIN_WARPS / 4);   // 16 columns per drain thread
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
static_assert(SMEM_BYTES <= 227 * 1024 && NLEV * BN <= 512, "shared memory, TMEM");

// ----------------------------------------------------------------- packing
struct DigitSide {
    const cplx* src;
    long long s_r, s_ki, s_ko, s_bi, s_bo;   // strides of row r, K (ki, ko), batch
    int R, Ki, Ko, Bi, Bo;
    int conj, embed;
    int Rpad;                                // rows per batch in the planes (complex)
    int Kc;                                  // padded complex K
    long long rows;                          // real rows in a plane
    uint16_t* planes;                        // ND planes of rows x 2 Kc bf16
    int* exps;                               // per complex row: biased exponent field of its largest entry
    uint16_t* mag;                           // rows x Kc bf16: max(|re|, |im|) 2^-E, rounded down; null: no check
    unsigned long long* l1;                  // per complex row: sum of (|re| + |im|) 2^-E in units of 2^-16
};

constexpr int PK_ROWS = 32, PK_THREADS = 256, PK_KT = 32;

__device__ __forceinline__ int exp_field(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); }

// Row f = b * Rpad + r of a side: base pointer, or null for padding.
__device__ __forceinline__ const cplx* row_base(const DigitSide& s, long long f) {
    const long long nrow = (long long)s.Rpad * s.Bi * s.Bo;
    if (f >= nrow) return nullptr;
    const long long b = f / s.Rpad;
    const int r = (int)(f - b * s.Rpad);
    if (r >= s.R) return nullptr;
    const int bi = (int)(b % s.Bi), bo = (int)(b / s.Bi);
    return s.src + bi * s.s_bi + bo * s.s_bo + r * s.s_r;
}

// Largest exponent field of 32 rows over K range [k0, k1) into mx[32]
// (zeroed by the caller): lanes run along whichever of row and K is the
// closer stride, so the gather is coalesced.
__device__ void max_exps(const DigitSide& s, const cplx* const* base, int k0, int k1, int* mx) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (s.s_r <= s.s_ki) {
        const cplx* p = base[lane];
        int m = 0;
        if (p)
            for (int k = k0 + warp; k < k1; k += PK_THREADS / 32) {
                const cplx v = p[(k % s.Ki) * s.s_ki + (k / s.Ki) * s.s_ko];
                m = max(m, max(exp_field(v.x), exp_field(v.y)));
            }
        atomicMax(&mx[lane], m);
    } else {
        for (int r = warp; r < PK_ROWS; r += PK_THREADS / 32) {
            const cplx* p = base[r];
            int m = 0;
            if (p)
                for (int k = k0 + lane; k < k1; k += 32) {
                    const cplx v = p[(k % s.Ki) * s.s_ki + (k / s.Ki) * s.s_ko];
                    m = max(m, max(exp_field(v.x), exp_field(v.y)));
                }
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) mx[r] = max(mx[r], m);
        }
    }
}

// x on the grid 2^(E - 55), E = emax - 1022: the integer t, round to nearest
// even, plus 128 in each of its six low bytes.  Byte i of the result minus 128
// is then the signed digit of weight 256^i, and bits 48.. the highest digit:
// one 64-bit addition carries for all of them.
__device__ __forceinline__ unsigned long long biased_digits(double x, int emax) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((u >> 52) & 0x7FF);
    unsigned long long m = u & 0xFFFFFFFFFFFFFULL;
    if (e) m |= 1ULL << 52;
    const int sh = max(e, 1) - max(emax, 1) + 2;
    if (sh >= 0) {
        m <<= sh;
    } else if (sh > -56) {
        const unsigned long long low = m & ((1ULL << -sh) - 1), half = 1ULL << (-sh - 1);
        m >>= -sh;
        if (low > half || (low == half && (m & 1))) ++m;
    } else {
        m = 0;
    }
    const long long t = (u >> 63) ? -(long long)m : (long long)m;
    return (unsigned long long)t + 0x808080808080ULL;
}

// Digit q (0 the highest) of biased digits t as a float: the byte under the
// exponent of 2^23, minus 2^23 + 128 (the highest digit through a conversion).
__device__ __forceinline__ float digit_float(unsigned long long t, int q) {
    if (q == 0) return (float)(int)((long long)t >> 48);
    const uint32_t w = q <= 2 ? (uint32_t)(t >> 32) : (uint32_t)t;
    const int byte = q <= 2 ? 2 - q : 6 - q;   // byte of the word
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440u | (uint32_t)byte)) - 8388736.0f;
}
// (lo, hi) as a bf16 pair: digits are integers up to 128, so the upper half of
// the float is exact.
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// max(|re|, |im|) 2^-E of an entry as bf16, rounded down; at least 2^-60 unless
// the entry is zero (a product of two is zero only if one of them is).
__device__ __forceinline__ uint16_t magnitude(cplx v, int emax) {
    const uint32_t hx = (uint32_t)__double2hiint(v.x) & 0x7FFFFFFFu, hy = (uint32_t)__double2hiint(v.y) & 0x7FFFFFFFu;
    const uint32_t h = hx > hy ? hx : hy;
    const int e = (int)(h >> 20), d = emax - e;
    if (e > 0 && d < 60) return (uint16_t)(((126 - d) << 7) | ((h >> 13) & 0x7Fu));
    return (h | (uint32_t)__double2loint(v.x) | (uint32_t)__double2loint(v.y)) ? (uint16_t)((126 - 59) << 7) : (uint16_t)0;
}
// |t| of biased digits in units of 2^39 (2^-16 of the row's largest), rounded up.
__device__ __forceinline__ unsigned l1_units(unsigned long long biased) {
    const long long t = (long long)(biased - 0x808080808080ULL);
    return (unsigned)(((t < 0 ? -t : t) + ((1LL << 39) - 1)) >> 39);
}

// Row exponents over blocks of K (long K only): exps and l1 zeroed before.
__global__ void __launch_bounds__(PK_THREADS) digit_max_kernel(DigitSide sp, DigitSide sq, int nbp, int kb,
                                                              const int* skip) {
    pdl_begin();
    if (skip && *(volatile const int*)skip) return;
    const DigitSide& s = (int)blockIdx.x < nbp ? sp : sq;
    const long long f0 = (long long)((int)blockIdx.x < nbp ? blockIdx.x : blockIdx.x - nbp) * PK_ROWS;
    __shared__ const cplx* base[PK_ROWS];
    __shared__ int mx[PK_ROWS];
    if (threadIdx.x < PK_ROWS) {
        base[threadIdx.x] = row_base(s, f0 + threadIdx.x);
        mx[threadIdx.x] = 0;
    }
    __syncthreads();
    const int K = s.Ki * s.Ko, k0 = blockIdx.y * kb;
    max_exps(s, base, k0, min(K, k0 + kb), mx);
    __syncthreads();
    if (threadIdx.x < PK_ROWS && base[threadIdx.x]) atomicMax(&s.exps[f0 + threadIdx.x], mx[threadIdx.x]);
}

// Digits of 32 rows over a block of K.  one_pass: this block sees the whole K
// and finds the exponents itself.
__global__ void __launch_bounds__(PK_THREADS) digit_pack_kernel(DigitSide sp, DigitSide sq, int nbp, int kb,
                                                               int one_pass, int* marked, const int* skip) {
    pdl_begin();
    if (skip && *(volatile const int*)skip) return;
    if (marked && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) marked[0] = marked[1] = 0;
    const bool isp = (int)blockIdx.x < nbp;
    const DigitSide& s = isp ? sp : sq;
    const long long f0 = (long long)(isp ? blockIdx.x : blockIdx.x - nbp) * PK_ROWS;
    __shared__ const cplx* base[PK_ROWS];
    __shared__ int mx[PK_ROWS];
    __shared__ cplx tile[PK_KT][PK_ROWS + 1];
    __shared__ unsigned long long l1[PK_ROWS];   // row r: added to by its own warp's lane 0 only
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long nrow = (long long)s.Rpad * s.Bi * s.Bo;
    if (threadIdx.x < PK_ROWS) {
        base[threadIdx.x] = row_base(s, f0 + threadIdx.x);
        mx[threadIdx.x] = 0;
        l1[threadIdx.x] = 0;
    }
    __syncthreads();
    const int K = s.Ki * s.Ko;
    if (one_pass) {
        max_exps(s, base, 0, K, mx);
        __syncthreads();
        if (threadIdx.x < PK_ROWS && f0 + threadIdx.x < nrow) s.exps[f0 + threadIdx.x] = mx[threadIdx.x];
    } else {
        if (threadIdx.x < PK_ROWS && f0 + threadIdx.x < nrow) mx[threadIdx.x] = s.exps[f0 + threadIdx.x];
    }
    __syncthreads();
    const int kend = min(s.Kc, (int)(blockIdx.y + 1) * kb);
    const long long plane = s.rows * 2LL * s.Kc;
    for (int k0 = blockIdx.y * kb; k0 < kend; k0 += PK_KT) {
        if (s.s_r <= s.s_ki) {
            const cplx* p = base[lane];
#pragma unroll
            for (int i = 0; i < PK_KT / 8; ++i) {
                const int kk = warp + 8 * i, k = k0 + kk;
                cplx v = make_double2(0.0, 0.0);
                if (p && k < K) v = p[(k % s.Ki) * s.s_ki + (k / s.Ki) * s.s_ko];
                tile[kk][lane] = v;
            }
        } else {
            const int k = k0 + lane;
            const long long off = (k % s.Ki) * s.s_ki + (k / s.Ki) * s.s_ko;
#pragma unroll
            for (int i = 0; i < PK_ROWS / 8; ++i) {
                const int r = warp + 8 * i;
                const cplx* p = base[r];
                cplx v = make_double2(0.0, 0.0);
                if (p && k < K) v = p[off];
                tile[lane][r] = v;
            }
        }
        __syncthreads();
        const int k = k0 + lane;
        for (int i = 0; i < PK_ROWS / 8; ++i) {
            const int r = warp + 8 * i;
            const long long f = f0 + r;
            if (f >= nrow) continue;
            unsigned l = 0;
            if (k < s.Kc) {
                uint16_t* o = s.planes + (s.embed ? 2 * f : f) * 2LL * s.Kc + 2LL * k;
                if (!base[r] || mx[r] == 0x7FF) {   // padding; rows with infinities or NaNs
#pragma unroll
                    for (int q = 0; q < ND; ++q) {
                        *reinterpret_cast<uint32_t*>(o + q * plane) = 0u;
                        if (s.embed) *reinterpret_cast<uint32_t*>(o + q * plane + 2LL * s.Kc) = 0u;
                    }
                    if (s.mag) s.mag[f * s.Kc + k] = 0;
                } else {
                    const cplx v = tile[lane][r];
                    const unsigned long long tr = biased_digits(v.x, mx[r]),
                                             ti = biased_digits(s.conj ? -v.y : v.y, mx[r]);
#pragma unroll
                    for (int q = 0; q < ND; ++q) {
                        const uint32_t w = bf16_pair(digit_float(tr, q), digit_float(ti, q));   // (re, im)
                        if (s.embed) {   // (re, -im) and (im, re)
                            *reinterpret_cast<uint32_t*>(o + q * plane) = w ^ 0x80000000u;
                            *reinterpret_cast<uint32_t*>(o + q * plane + 2LL * s.Kc) = __byte_perm(w, 0u, 0x1032);
                        } else {
                            *reinterpret_cast<uint32_t*>(o + q * plane) = w;
                        }
                    }
                    if (s.mag) {
                        s.mag[f * s.Kc + k] = magnitude(v, mx[r]);
                        l = l1_units(tr) + l1_units(ti);
                    }
                }
            }
            if (s.mag) {
                l = __reduce_add_sync(0xffffffffu, l);
                if (lane == 0) l1[r] += l;
            }
        }
        __syncthreads();
    }
    if (s.mag && threadIdx.x < PK_ROWS && f0 + threadIdx.x < nrow) {
        if (gridDim.y == 1) s.l1[f0 + threadIdx.x] = l1[threadIdx.x];
        else atomicAdd(&s.l1[f0 + threadIdx.x], l1[threadIdx.x]);
    }
}

// ---------------------------------------------------------------- the GEMM
struct DigitGemm {
    GemmArgs g;                  // strides, alpha, beta; the operands for rows with infinities or NaNs
    int swapped;                 // P = the B side (columns n of C)
    int Pn, Qn;                  // valid complex rows per batch
    int Pp, Qp;                  // padded rows per batch: complex P rows, real Q rows
    int p_vbi, p_vbo, q_vbi, q_vbo;
    int nst;                     // K' / BK
    int n_ptiles, n_qtiles, batches;
    int q_fast;
    int nsplit, cps;             // K ranges per tile, chunks per range
    const int* expP;             // 0x7FF: the row holds an infinity or a NaN
    const int* expQ;
    // outputs left to digit_fix_kernel, null: none; bit i of word ((b n_qtiles +
    // qt) Pp + p): complex Q row 32 qt + i
    uint32_t* mask;
    int* marked;                 // [0] how many, [1] in how many words
    uint32_t* list;              // those words, in any order
    const uint16_t *magP, *magQ;
    const unsigned long long *l1P, *l1Q;
    int Kc;
    unsigned long long stall_ns; // test hook: > 0 makes the drain warps wait this long on a barrier that nothing arrives at
    cplx* W;                     // partial sums of split K (layout of splitk_f64_kernel)
    int* err;
    const int* skip;             // not null and set: nothing to do
};

// 64-byte swizzle, K-major, 8-row groups 512 bytes apart; the address (lower
// word) varies.
constexpr uint32_t DESC_HI = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr & 0x3FFFF) >> 4) | (1u << 16); }

// D = F32, A = B = BF16, K-major, M = 128, N = 64.
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t dt, uint32_t a, uint32_t b, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %4, 0;\n mov.b64 da, {%1, %5};\n mov.b64 db, {%2, %5};\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}\n" ::"r"(dt),
        "r"(a), "r"(b), "r"(IDESC), "r"(acc), "r"(DESC_HI));
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// (h 2^32 + lo) 2^sc as a double, rounded once (to nearest even); results
// outside the normal range go through scalbn.
__device__ __forceinline__ double to_double(long long h, long long lo, int sc) {
    h += lo >> 32;
    unsigned l = (unsigned)lo;
    const bool neg = h < 0;
    if (neg) {
        h = ~h;
        l = ~l;
        if (++l == 0) ++h;
    }
    if (h == 0 && l == 0) return 0.0;
    unsigned long long uh = (unsigned long long)h, top;
    int lz = uh ? __clzll((long long)uh) : 64 + __clz((int)l);   // zeros before the first bit, of 96
    unsigned sticky = 0;
    if (lz >= 64) {
        top = (unsigned long long)l << (lz - 32);
    } else if (lz >= 32) {
        top = (uh << lz) | ((unsigned long long)l << (lz - 32));
    } else if (lz > 0) {
        top = (uh << lz) | (l >> (32 - lz));
        sticky = l << lz;
    } else {
        top = uh;
        sticky = l;
    }
    unsigned long long mant = top >> 11;
    const unsigned rem = (unsigned)top & 0x7FFu;
    if (rem > 0x400u || (rem == 0x400u && (sticky || (mant & 1)))) ++mant;
    const unsigned long long sgn = neg ? 1ULL << 63 : 0ULL;
    const int e = 95 - lz + 1023;           // field of the leading bit before scaling
    const int es = e + sc;
    if (es > 0 && es < 2046)
        return __longlong_as_double((long long)(sgn | ((((unsigned long long)es) << 52) + (mant - (1ULL << 52)))));
    const double d = __longlong_as_double((long long)(sgn | ((((unsigned long long)e) << 52) + (mant - (1ULL << 52)))));
    return scalbn(d, sc);
}

// Plane row (complex P rows, real Q rows) where batch b starts.
__device__ __forceinline__ int first_row(const DigitGemm& ea, int b, int vbi, int vbo, int pad) {
    const int bi = b % ea.g.Bi, bo = b / ea.g.Bi;
    return ((vbi ? bi : 0) + (vbo ? bo * (vbi ? ea.g.Bi : 1) : 0)) * pad;
}

__device__ __forceinline__ void store_output(const DigitGemm& ea, int m, int n, int bi, int bo, cplx r) {
    const GemmArgs& g = ea.g;
    cplx* cp = g.C + bi * g.c_bi + bo * g.c_bo + m * g.c_m + n * g.c_n;
    if (!(g.alpha.x == 1.0 && g.alpha.y == 0.0)) {
        const cplx v = r;
        r.x = g.alpha.x * v.x - g.alpha.y * v.y;
        r.y = g.alpha.x * v.y + g.alpha.y * v.x;
    }
    if (!(g.beta.x == 0.0 && g.beta.y == 0.0)) {
        const cplx o = *cp;
        if (g.beta.x == 1.0 && g.beta.y == 0.0) {
            r.x += o.x;
            r.y += o.y;
        } else {
            r.x += g.beta.x * o.x - g.beta.y * o.y;
            r.y += g.beta.x * o.y + g.beta.y * o.x;
        }
    }
    *cp = r;
}

// --------------------------------------------------------------- the check
// S = sum_k max(|re|, |im|)_p max(|re|, |im|)_q 2^-(Ep + Eq), at most
// sum |p_k||q_k| in those units, for 32 x 32 outputs per warp.  With l the l1
// sums, the digits' error is below 2^-56 (l_p + l_q) + K 2^-60 and an FMA chain's
// bound is 2 K 2^-53 S: marked is what has S < (l_p + l_q) / (16 K) + 2^-8, except
// S = 0 (every product zero, and so is the digits' result), and rows with
// infinities or NaNs.  Operands of one size reach the threshold within the
// first few dozen K and stop there: only graded and sparse rows are summed to
// the end.  For a long K and few outputs that is a chain of loads (128 x 128 x
// 16384: 390 us with a warp per 32 x 32 tile), so there (LONG) one of a block's 4
// warps looks at the first 128 K, and if that is not enough all of them share
// the tile's K, load ahead, and add their sums in a fixed order (109 us; the
// step below 1.83 -> 1.74 s).  The order of K is free, so a lane loads 16 bytes of a
// row and feeds them to two k16 steps.
constexpr int CK_WARPS = 4, CK_THREADS = 32 * CK_WARPS;
template <bool LONG>
__global__ void __launch_bounds__(CK_THREADS) digit_check_kernel(DigitGemm ea) {
    pdl_begin();
    __shared__ float sums[LONG ? CK_WARPS : 1][32][32];   // [warp][accumulator][lane]
    __shared__ int s_more;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nqc = ea.n_qtiles, npc = ea.Pp / 32;   // 32 x 32 outputs per warp (LONG: per block)
    const long long tile = LONG ? blockIdx.x : (long long)blockIdx.x * CK_WARPS + warp;
    if (tile >= (long long)npc * nqc * ea.batches) return;
    const int b = (int)(tile / (npc * nqc)), rest = (int)(tile % (npc * nqc));
    const int p0 = rest % npc * 32, qt = rest / npc, q0 = qt * 32;
    const long long prow = first_row(ea, b, ea.p_vbi, ea.p_vbo, ea.Pp) + p0;
    const long long qrow = first_row(ea, b, ea.q_vbi, ea.q_vbo, ea.Qp) / 2 + q0;
    const int g8 = lane >> 2, j4 = lane & 3;
    const float c1 = 1.01f / (16.0f * 65536.0f * (float)(ea.g.Ki * ea.g.Ko));
    float lp[4], lq[8];                        // thresholds' parts: rows g8 + 8 i, columns 8 i + 2 j4 and + 1
    bool pbad[4], qbad[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        lp[i] = 0.00391f + c1 * (float)ea.l1P[prow + g8 + 8 * i];
        pbad[i] = ea.expP[prow + g8 + 8 * i] == 0x7FF;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int c = 8 * (i >> 1) + 2 * j4 + (i & 1);
        lq[i] = c1 * (float)ea.l1Q[qrow + c];
        qbad[i] = ea.expQ[qrow + c] == 0x7FF;
    }
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    // marks of this lane: row i (g8 + 8 i), column c (8 (c >> 1) + 2 j4 + (c & 1))
    auto marks = [&](bool final) {
        unsigned out[4] = {0u, 0u, 0u, 0u}, any = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float S = acc[i >> 1][c >> 1][(i & 1) * 2 + (c & 1)];
                const bool valid = p0 + g8 + 8 * i < ea.Pn && q0 + 8 * (c >> 1) + 2 * j4 + (c & 1) < ea.Qn;
                const bool low = S < lp[i] + lq[c] && !(final && S == 0.f);
                if (valid && (low || (final && (pbad[i] || qbad[c])))) out[i] |= 1u << (8 * (c >> 1) + 2 * j4 + (c & 1));
            }
#pragma unroll
        for (int i = 0; i < 4; ++i) any |= out[i];
        if (final) {
            unsigned n = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                unsigned w = out[i];
                w |= __shfl_xor_sync(0xffffffffu, w, 1);
                w |= __shfl_xor_sync(0xffffffffu, w, 2);
                if (j4 == 0) {
                    const long long word = ((long long)b * nqc + qt) * ea.Pp + p0 + g8 + 8 * i;
                    ea.mask[word] = w;
                    if (w) ea.list[atomicAdd(ea.marked + 1, 1)] = (uint32_t)word;
                    n += __popc(w);
                }
            }
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0 && n) atomicAdd(ea.marked, (int)n);
        }
        return any != 0;
    };
    const uint16_t* mp = ea.magP + (prow + g8) * ea.Kc;
    const uint16_t* mq = ea.magQ + (qrow + g8) * ea.Kc;
    uint4 a[4], bq[4];
    auto load = [&](int slice, uint4* x, uint4* y) {   // 32 K of every row
        const int k = 32 * slice + 8 * j4;
        const bool in = k < ea.Kc;             // Kc is a multiple of 16
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[i] = in ? *reinterpret_cast<const uint4*>(mp + 8LL * i * ea.Kc + k) : make_uint4(0, 0, 0, 0);
            y[i] = in ? *reinterpret_cast<const uint4*>(mq + 8LL * i * ea.Kc + k) : make_uint4(0, 0, 0, 0);
        }
    };
    auto multiply = [&] {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float* d = acc[i][j];
                asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                             : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                             : "r"(a[2 * i].x), "r"(a[2 * i + 1].x), "r"(a[2 * i].y), "r"(a[2 * i + 1].y), "r"(bq[j].x), "r"(bq[j].y));
                asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                             : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                             : "r"(a[2 * i].z), "r"(a[2 * i + 1].z), "r"(a[2 * i].w), "r"(a[2 * i + 1].w), "r"(bq[j].z), "r"(bq[j].w));
            }
    };
    const int slices = (ea.Kc + 31) / 32;
    auto sum_slices = [&](int first, int step, bool stop) {   // the next one in flight
        uint4 an[4], bn[4];
        load(first, a, bq);
        for (int it = first; it < slices; it += step) {
            load(it + step, an, bn);
            multiply();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = an[i];
                bq[i] = bn[i];
            }
            if (stop && (it & 3) == 3 && !__any_sync(0xffffffffu, marks(false))) break;
        }
    };
    if (!LONG) {
        sum_slices(0, 1, true);
        marks(true);
        return;
    }
    if (warp == 0) {   // are the first four slices enough?
        for (int it = 0; it < 4; ++it) {
            load(it, a, bq);
            multiply();
        }
        const bool more = __any_sync(0xffffffffu, marks(false));
        if (lane == 0) s_more = more;
    }
    __syncthreads();
    if (s_more) {
        float* d = &acc[0][0][0];
#pragma unroll
        for (int i = 0; i < 32; ++i) d[i] = 0.f;
        sum_slices(warp, CK_WARPS, false);
#pragma unroll
        for (int i = 0; i < 32; ++i) sums[warp][i][lane] = d[i];
        __syncthreads();
        if (warp == 0)
#pragma unroll
            for (int i = 0; i < 32; ++i)
                for (int w = 1; w < CK_WARPS; ++w) d[i] += sums[w][i][lane];
    }
    if (warp == 0) marks(true);
}

// sum over k in [k0, k1) of A_k B_k, one FMA chain.
__device__ __forceinline__ cplx fma_chain(const GemmArgs& g, const cplx* A0, const cplx* B0, int k0, int k1) {
    cplx s = make_double2(0.0, 0.0);
    int ki = k0 % g.Ki, ko = k0 / g.Ki;
    while (k0 < k1) {
        const int run = min(g.Ki - ki, k1 - k0);
        const cplx* A = A0 + ki * g.a_ki + ko * g.a_ko;
        const cplx* B = B0 + ki * g.b_ki + ko * g.b_ko;
#pragma unroll 4
        for (int i = 0; i < run; ++i) {
            cplx a = *A, v = *B;
            if (g.conjA) a.y = -a.y;
            if (g.conjB) v.y = -v.y;
            s.x = fma(a.x, v.x, s.x);
            s.x = fma(-a.y, v.y, s.x);
            s.y = fma(a.x, v.y, s.y);
            s.y = fma(a.y, v.x, s.y);
            A += g.a_ki;
            B += g.b_ki;
        }
        k0 += run;
        ki = 0;
        ++ko;
    }
    return s;
}

// A marked output's value to where the digits' would have gone.
__device__ __forceinline__ void store_marked(const DigitGemm& ea, int m, int n, int b, cplx s) {
    if (ea.nsplit > 1) {   // the whole sum in the first range's place
        for (int ks = 0; ks < ea.nsplit; ++ks)
            ea.W[(((long long)ks * ea.batches + b) * ea.g.N + n) * ea.g.M + m] = ks ? make_double2(0.0, 0.0) : s;
    } else {
        store_output(ea, m, n, b % ea.g.Bi, b / ea.g.Bi, s);
    }
}

// The marked outputs in plain FP64.
// Few are marked, often of a long K: the words that hold any are spread over the
// SMs, each to W warps, as many as there are warps for (1 to all 8 of a block),
// and a word's outputs share its 32 W lanes, each with a slice of K.
// Many (an eighth and more: operands graded against each other): 32 outputs side
// by side, one per lane, to a warp, or where there are too few of these for two
// warps each, to a block whose 8 warps take a slice of K each, as the direct
// kernel of gemm_f64.cu does (all marked, whole call: 16384 x 128 x 128 3.6 ms by
// words, 3.3 so, 2.1 by the direct kernel; 128 x 128 x 16384 17.3, 4.0, 2.2).
// Slices are added in order.
// Measured, a step of 8x8, chi = 128 from a product state, 0.01 to 2 % of
// the outputs of its K = 10368 and 16384 contractions marked: 2.90 s with
// 256 words to a block wherever their marked outputs lie, 1.83 s so.
constexpr int FX_THREADS = 256, FX_WARPS = FX_THREADS / 32;
__global__ void __launch_bounds__(FX_THREADS) digit_fix_kernel(DigitGemm ea) {
    pdl_begin();
    const int nwords = *(volatile int*)(ea.marked + 1);
    if (nwords == 0) return;
    __shared__ cplx part[FX_WARPS][32];
    const GemmArgs& g = ea.g;
    const int K = g.Ki * g.Ko, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (8LL * *(volatile int*)ea.marked >= (long long)g.M * g.N * ea.batches) {
        const int mb = (g.M + 31) / 32;
        const long long groups = (long long)mb * g.N * ea.batches;
        const int S = groups < 2LL * gridDim.x * FX_WARPS ? FX_WARPS : 1, kc = (K + S - 1) / S;   // slices of K
        const int slice = warp % S;
        for (long long i = blockIdx.x * (FX_WARPS / S) + warp / S; i < groups; i += (long long)gridDim.x * (FX_WARPS / S)) {
            const int m = (int)(i % mb) * 32 + lane;
            const long long r = i / mb;
            const int n = (int)(r % g.N), b = (int)(r / g.N), p = ea.swapped ? n : m, q = ea.swapped ? m : n;
            const bool mine = m < g.M && ((ea.mask[((long long)b * ea.n_qtiles + (q >> 5)) * ea.Pp + p] >> (q & 31)) & 1u);
            if (!__any_sync(0xffffffffu, mine)) continue;   // S > 1: the same in every warp of the block
            cplx s = make_double2(0.0, 0.0);
            if (mine)
                s = fma_chain(g, g.A + (b % g.Bi) * g.a_bi + (b / g.Bi) * g.a_bo + m * g.a_m,
                              g.B + (b % g.Bi) * g.b_bi + (b / g.Bi) * g.b_bo + n * g.b_n, min(K, slice * kc),
                              min(K, (slice + 1) * kc));
            if (S > 1) {
                part[warp][lane] = s;
                __syncthreads();
                if (warp == 0)
                    for (int w = 1; w < S; ++w) {
                        s.x += part[w][lane].x;
                        s.y += part[w][lane].y;
                    }
                __syncthreads();
            }
            if (mine && slice == 0) store_marked(ea, m, n, b, s);
        }
        return;
    }
    int W = 1;
    while (W < FX_WARPS && (long long)nwords * W * 2 <= (long long)gridDim.x * FX_WARPS) W *= 2;
    const int per = FX_WARPS / W, grp = warp / W, t = (int)threadIdx.x % (32 * W);
    for (long long i0 = (long long)blockIdx.x * per; i0 < nwords; i0 += (long long)gridDim.x * per) {
        const bool on = i0 + grp < nwords;
        const uint32_t word = on ? ea.list[i0 + grp] : 0u;
        uint32_t w = on ? ea.mask[word] : 0u;
        const int n = max(1, __popc(w));
        int L = W;                              // n <= 32: lanes per output
        while (n * L * 2 <= 32 * W) L *= 2;
        const int o = t / L;                    // output of the word
        const bool mine = o < __popc(w);
        cplx s = make_double2(0.0, 0.0);
        int m = 0, nn = 0, b = 0;
        if (mine) {
            for (int i = 0; i < o; ++i) w &= w - 1;
            const int p = (int)(word % (uint32_t)ea.Pp), rest = (int)(word / (uint32_t)ea.Pp);
            const int q = rest % ea.n_qtiles * 32 + __ffs((int)w) - 1;
            b = rest / ea.n_qtiles;
            m = ea.swapped ? q : p;
            nn = ea.swapped ? p : q;
            const int kc = (K + L - 1) / L;
            s = fma_chain(g, g.A + (b % g.Bi) * g.a_bi + (b / g.Bi) * g.a_bo + m * g.a_m,
                          g.B + (b % g.Bi) * g.b_bi + (b / g.Bi) * g.b_bo + nn * g.b_n, min(K, t % L * kc),
                          min(K, (t % L + 1) * kc));
        }
        for (int d = min(L, 32) / 2; d > 0; d /= 2) {   // a warp has one L
            s.x += __shfl_xor_sync(0xffffffffu, s.x, d);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, d);
        }
        if (W > 1) {   // L > 32: the warps of an output
            __syncthreads();
            if (lane == 0) part[warp][0] = s;
            __syncthreads();
            if (mine && t % L == 0)
                for (int i = 1; i < L / 32; ++i) {
                    s.x += part[warp + i][0].x;
                    s.y += part[warp + i][0].y;
                }
        }
        if (mine && t % L == 0) store_marked(ea, m, nn, b, s);
    }
}

__global__ void __launch_bounds__(THREADS, 1)
    digit_gemm_kernel(const __grid_constant__ CUtensorMap mP, const __grid_constant__ CUtensorMap mQ, DigitGemm ea) {
    pdl_wait();
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* lfull = empty + STAGES;      // [NLEV] level accumulated
    uint64_t* lempty = lfull + NLEV;       // [NLEV] level drained
    uint64_t* mdone = lempty + NLEV;
    uint64_t* stallbar = mdone + 1;        // test hook: never arrived at
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(stallbar + 1);

    // an earlier launch on this workspace gave up (the host reports the error at
    // its next check), or the caller's flag is set: do nothing
    __shared__ int s_skip, s_marked;
    if (threadIdx.x == 0) {
        s_skip = *(volatile int*)ea.err || (ea.skip && *(volatile const int*)ea.skip);
        s_marked = ea.mask && *(volatile int*)ea.marked;
    }
    __syncthreads();
    if (s_skip) return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long grid_tiles = (long long)ea.n_ptiles * ea.n_qtiles;
    const long long ntiles = grid_tiles * ea.batches * ea.nsplit;
    auto tile_of = [&](long long t, int& pt, int& qt, int& b, int& ks) {
        const long long w = t % grid_tiles, rest = t / grid_tiles;
        if (ea.q_fast) {
            qt = (int)(w % ea.n_qtiles);
            pt = (int)(w / ea.n_qtiles);
        } else {
            pt = (int)(w % ea.n_ptiles);
            qt = (int)(w / ea.n_ptiles);
        }
        b = (int)(rest % ea.batches);
        ks = (int)(rest / ea.batches);
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < NLEV; ++i) {
            mbar_init(&lfull[i], 1);
            mbar_init(&lempty[i], DRAIN_THREADS);
        }
        mbar_init(mdone, 1);
        mbar_init(stallbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(NLEV * BN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == TMA_WARP) {
        if (lane == 0) {
            unsigned it = 0;
            bool ok = true;
            for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                int pt, qt, b, ks;
                tile_of(t, pt, qt, b, ks);
                const int prow = first_row(ea, b, ea.p_vbi, ea.p_vbo, ea.Pp) + pt * BM;
                const int qrow = first_row(ea, b, ea.q_vbi, ea.q_vbo, ea.Qp) + qt * BN;
                const int st0 = ks * ea.cps * CHUNK_ST, st1 = min(ea.nst, (ks + 1) * ea.cps * CHUNK_ST);
                for (int st = st0; st < st1; ++st, ++it) {
                    const unsigned s = it % STAGES, round = it / STAGES;
                    if (it >= STAGES && !mbar_wait(&empty[s], (round - 1) & 1, ea.err)) {
                        ok = false;
                        break;
                    }
                    uint8_t* p = smem + s * STAGE_BYTES;
                    mbar_expect_tx(&full[s], STAGE_BYTES);
                    tma_load_3d(p, &mP, &full[s], st * BK, prow, 0);
                    tma_load_3d(p + P_BYTES, &mQ, &full[s], st * BK, qrow, 0);
                }
            }
            // wait for loads that the MMA issuer did not consume
            for (unsigned i = it > STAGES ? it - STAGES : 0; i < it; ++i)
                mbar_drain(&full[i % STAGES], (i / STAGES) & 1);
        }
        __syncwarp();
    } else if (warp == MMA_WARP) {
        // the whole warp walks the loop, one elected lane issues: unrolled, the
        // descriptors are immediate offsets from uniform registers (a loop over the
        // digits took 110 clk per MMA to issue, unrolled in one lane's branch 70; the
        // MMA takes 32 to 48).  Uniform: 128 x 128 x 16384 204 -> 187 us, 4096 x 64 x 64
        // in batches of 4 61 -> 55 us.
        const uint32_t lo0 = desc_lo(smem_u32(smem));
        unsigned it = 0, cg = 0;
        bool ok = true;
        for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            const int ks = (int)(t / (grid_tiles * ea.batches));
            const int st1 = min(ea.nst, (ks + 1) * ea.cps * CHUNK_ST);
            for (int c0 = ks * ea.cps * CHUNK_ST; c0 < st1 && ok; c0 += CHUNK_ST, ++cg) {
                const int c1 = min(st1, c0 + CHUNK_ST);
                for (int st = c0; st < c1 && ok; ++st, ++it) {
                    const unsigned s = it % STAGES, round = it / STAGES;
                    if (!__all_sync(0xffffffffu, mbar_wait(&full[s], round & 1, ea.err))) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t dp = lo0 + s * (STAGE_BYTES >> 4), dq = dp + (P_BYTES >> 4);
#pragma unroll
                    for (int l = 0; l < NLEV; ++l) {
                        if (!ok) break;
                        if (st == c0 && cg > 0) {
                            if (!__all_sync(0xffffffffu, mbar_wait(&lempty[l], (cg - 1) & 1, ea.err))) {
                                ok = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        }
                        const int i0 = l > ND - 1 ? l - (ND - 1) : 0, i1 = l < ND - 1 ? l : ND - 1;
                        if (elect_one()) {
#pragma unroll
                            for (int i = i0; i <= i1; ++i) {
                                const uint32_t a = dp + (i * P_PLANE >> 4), q = dq + ((l - i) * Q_PLANE >> 4);
                                mma_bf16(tmem + l * BN, a, q, (st > c0 || i > i0) ? 1u : 0u);
                                mma_bf16(tmem + l * BN, a + 2, q + 2, 1u);   // 16 bf16 = 32 bytes along K
                            }
                            if (st == c1 - 1) mma_commit(&lfull[l]);
                        }
                        __syncwarp();
                    }
                    if (elect_one()) mma_commit(&empty[s]);
                    __syncwarp();
                }
            }
        }
        if (elect_one()) mma_commit(mdone);
        __syncwarp();
        mbar_drain(mdone, 0);
        __syncwarp();
    } else {
        const int quad = warp & 3, col0 = (warp >> 2) * DCOLS;
        unsigned cg = 0;
        bool ok = true;
        // test hook: the other roles see the error flag and abort as after a real timeout
        if (ea.stall_ns > 0 && !__all_sync(0xffffffffu, mbar_wait(stallbar, 0, ea.err, ea.stall_ns))) ok = false;
        for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            int pt, qt, b, ks;
            tile_of(t, pt, qt, b, ks);
            const int st0 = ks * ea.cps * CHUNK_ST, st1 = min(ea.nst, (ks + 1) * ea.cps * CHUNK_ST);
            long long sh[DCOLS], sl[DCOLS];   // levels 0-3 and 4-7, in units of 2^32 and 1
#pragma unroll
            for (int j = 0; j < DCOLS; ++j) sh[j] = sl[j] = 0;
            for (int c0 = st0; c0 < st1 && ok; c0 += CHUNK_ST, ++cg) {
#pragma unroll
                for (int l = 0; l < NLEV; ++l) {
                    if (!ok) break;
                    if (!__all_sync(0xffffffffu, mbar_wait(&lfull[l], cg & 1, ea.err))) {   // warp-uniform
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (int h = 0; h < DCOLS; h += 8) {
                        uint32_t v[8];
                        tmem_ld8(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(l * BN + col0 + h), v);
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const long long w = (long long)__float2int_rn(__uint_as_float(v[j])) * (1 << (8 * (3 - (l & 3))));
                            if (l < 4) sh[h + j] += w;
                            else sl[h + j] += w;
                        }
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&lempty[l])) : "memory");
                }
            }
            if (!ok) break;
            const int p = pt * BM + quad * 32 + lane;
            if (p < ea.Pn) {
                const int bi = b % ea.g.Bi, bo = b / ea.g.Bi;
                const int ep = ea.expP[first_row(ea, b, ea.p_vbi, ea.p_vbo, ea.Pp) + p];
                const int* eq = ea.expQ + first_row(ea, b, ea.q_vbi, ea.q_vbo, ea.Qp) / 2;
                const uint32_t left = s_marked ? ea.mask[((long long)b * ea.n_qtiles + qt) * ea.Pp + p] >> (col0 >> 1) : 0u;
#pragma unroll
                for (int j = 0; j < DCOLS; j += 2) {
                    const int q = (qt * BN + col0 + j) >> 1;
                    if (q >= ea.Qn || ((left >> (j >> 1)) & 1u)) continue;
                    const int e = eq[q];
                    const int m = ea.swapped ? q : p, n = ea.swapped ? p : q;
                    cplx r;
                    if (ep == 0x7FF || e == 0x7FF) {   // only without the check
                        r = make_double2(CUDART_NAN, CUDART_NAN);
                    } else {
                        const int sc = max(ep, 1) + max(e, 1) - 2 * 1022 - 70;   // E_p + E_q - 110 + 40
                        r = make_double2(to_double(sh[j], sl[j], sc), to_double(sh[j + 1], sl[j + 1], sc));
                    }
                    if (ea.nsplit > 1) ea.W[(((long long)ks * ea.batches + b) * ea.g.N + n) * ea.g.M + m] = r;
                    else store_output(ea, m, n, bi, bo, r);
                }
            }
            __syncwarp();
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(NLEV * BN));
    }
}

// ------------------------------------------------------------------- host
constexpr int N_SM = 152;
constexpr long long MAX_PLANE_BYTES = 1LL << 30;   // planes of one launch; larger batches run in parts

inline long long round_up(long long x, long long m) { return (x + m - 1) / m * m; }

struct DPlan {
    bool ok = false;
    DigitGemm d{};
    long long np = 0, nq = 0;             // packed batches of P and Q
    int Kp = 0;
    size_t p_off = 0, q_off = 0, ep_off = 0, eq_off = 0, lp_off = 0, lq_off = 0, mp_off = 0, mq_off = 0, mask_off = 0, list_off = 0, w_off = 0, bytes = 0;
};

DPlan plan(const GemmArgs& g, bool elementwise) {
    DPlan pl;
    const long long K = (long long)g.Ki * g.Ko;
    if (g.M <= 0 || g.N <= 0 || K <= 0 || g.Bi <= 0 || g.Bo <= 0) return pl;
    DigitGemm& d = pl.d;
    d.g = g;
    const int a_vbi = g.a_bi != 0 && g.Bi > 1, a_vbo = g.a_bo != 0 && g.Bo > 1;
    const int b_vbi = g.b_bi != 0 && g.Bi > 1, b_vbo = g.b_bo != 0 && g.Bo > 1;
    const long long na = (a_vbi ? g.Bi : 1) * (long long)(a_vbo ? g.Bo : 1);
    const long long nb = (b_vbi ? g.Bi : 1) * (long long)(b_vbo ? g.Bo : 1);
    // P: the side that gives fewer 128 x 32 tiles, then fewer packed rows
    auto tiles = [](long long p, long long q) { return round_up(p, BM) / BM * (round_up(2 * q, BN) / BN); };
    const long long ta = tiles(g.M, g.N), tb = tiles(g.N, g.M);
    d.swapped = tb < ta || (tb == ta && g.N * nb + 2LL * g.M * na < g.M * na + 2LL * g.N * nb);
    d.Pn = d.swapped ? g.N : g.M;
    d.Qn = d.swapped ? g.M : g.N;
    d.Pp = (int)round_up(d.Pn, BM);
    d.Qp = (int)round_up(2LL * d.Qn, BN);
    d.p_vbi = d.swapped ? b_vbi : a_vbi;
    d.p_vbo = d.swapped ? b_vbo : a_vbo;
    d.q_vbi = d.swapped ? a_vbi : b_vbi;
    d.q_vbo = d.swapped ? a_vbo : b_vbo;
    pl.np = d.swapped ? nb : na;
    pl.nq = d.swapped ? na : nb;
    pl.Kp = (int)round_up(2 * K, BK);
    d.nst = pl.Kp / BK;
    d.n_ptiles = d.Pp / BM;
    d.n_qtiles = d.Qp / BN;
    d.q_fast = d.n_qtiles < d.n_ptiles;
    d.batches = g.Bi * g.Bo;
    const long long t = (long long)d.n_ptiles * d.n_qtiles * d.batches;
    // split K: the number of ranges that minimises waves x (chunks + 1)
    const int nchunk = (d.nst + CHUNK_ST - 1) / CHUNK_ST;
    d.nsplit = 1;
    d.cps = nchunk;
    long long best = (t + N_SM - 1) / N_SM * (nchunk + 1);
    for (int n = 2; n <= std::min(nchunk, N_SM); ++n) {
        const int c = (nchunk + n - 1) / n, k = (nchunk + c - 1) / c;
        const long long cost = (t * k + N_SM - 1) / N_SM * (c + 1) + 1;
        if (cost < best) {
            best = cost;
            d.nsplit = k;
            d.cps = c;
        }
    }
    size_t off = 256;
    auto take = [&](size_t n) {
        const size_t o = off;
        off += (n + 255) / 256 * 256;
        return o;
    };
    pl.ep_off = take(sizeof(int) * pl.np * d.Pp);
    pl.eq_off = take(sizeof(int) * pl.nq * (d.Qp / 2));
    if (elementwise) {
        pl.lp_off = take(sizeof(unsigned long long) * pl.np * d.Pp);
        pl.lq_off = take(sizeof(unsigned long long) * pl.nq * (d.Qp / 2));
    }
    pl.p_off = take((size_t)ND * pl.np * d.Pp * pl.Kp * 2);
    pl.q_off = take((size_t)ND * pl.nq * d.Qp * pl.Kp * 2);
    d.Kc = pl.Kp / 2;
    if (elementwise) {
        pl.mp_off = take((size_t)pl.np * d.Pp * d.Kc * 2);
        pl.mq_off = take((size_t)pl.nq * (d.Qp / 2) * d.Kc * 2);
        pl.mask_off = take(sizeof(uint32_t) * (size_t)d.batches * d.n_qtiles * d.Pp);
        pl.list_off = take(sizeof(uint32_t) * (size_t)d.batches * d.n_qtiles * d.Pp);
    }
    if (d.nsplit > 1) pl.w_off = take((size_t)d.nsplit * d.batches * g.M * (size_t)g.N * sizeof(cplx));
    pl.bytes = off;
    pl.ok = pl.np * d.Pp < (1LL << 31) && pl.nq * d.Qp < (1LL << 31) &&
            (long long)d.batches * d.n_qtiles * d.Pp < (1LL << 31);   // words of the mask
    return pl;
}

bool make_map3(CUtensorMap* m, const void* base, long long rows, int kp, int box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)kp, (cuuint64_t)rows, (cuuint64_t)ND};
    cuuint64_t strides[2] = {(cuuint64_t)kp * 2, (cuuint64_t)kp * 2 * rows};
    cuuint32_t box[3] = {BK, (cuuint32_t)box_rows, ND};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The contraction in parts of at most MAX_PLANE_BYTES of planes, over the
// outer batch, then the inner one.
bool halve(const GemmArgs& g, GemmArgs& lo, GemmArgs& hi) {
    lo = hi = g;
    if (g.Bo > 1) {
        lo.Bo = g.Bo / 2;
        hi.Bo = g.Bo - lo.Bo;
        hi.A += lo.Bo * g.a_bo;
        hi.B += lo.Bo * g.b_bo;
        hi.C += lo.Bo * g.c_bo;
        return true;
    }
    if (g.Bi > 1) {
        lo.Bi = g.Bi / 2;
        hi.Bi = g.Bi - lo.Bi;
        hi.A += lo.Bi * g.a_bi;
        hi.B += lo.Bi * g.b_bi;
        hi.C += lo.Bi * g.c_bi;
        return true;
    }
    return false;
}

}  // namespace

// Rule: digits pay once the FP64 pipe would take longer than the fixed cost
// of packing and checking both sides plus the tile work (measured at the border:
// 4096 x 64 x 64 280 us on the FP64 pipe, 55 in digits; 64 x 64 x 64 9 us and 20).
bool digits_wanted(const GemmArgs& g) {
    const double K = (double)g.Ki * g.Ko, macs = (double)g.M * g.N * K * g.Bi * (double)g.Bo;
    if (std::min(g.M, g.N) < 16 || std::max(g.M, g.N) < 32 || K < 16) return false;
    DPlan pl = plan(g, true);
    if (!pl.ok || !encode_fn()) return false;
    const double f64_us = 4.0 + 8.0 * macs / 1.0e6;
    const double chunks = (double)pl.d.n_ptiles * pl.d.n_qtiles * pl.d.batches * ((pl.d.nst + CHUNK_ST - 1) / CHUNK_ST);
    const double us = 23.0 + 6.5 * std::max(1.0, chunks / N_SM) + (double)pl.bytes / 2.0e6;
    return us < f64_us;
}

size_t digits_workspace_bytes(const GemmArgs& g, bool elementwise) {
    DPlan pl = plan(g, elementwise);
    if (!pl.ok) return 0;
    if ((long long)pl.bytes > MAX_PLANE_BYTES) {
        GemmArgs lo, hi;
        if (halve(g, lo, hi)) return std::max(digits_workspace_bytes(lo, elementwise), digits_workspace_bytes(hi, elementwise));
    }
    return pl.bytes;
}

int launch_zgemm_digits(const GemmArgs& g, bool elementwise, cudaStream_t stream, void* workspace,
                        size_t workspace_bytes, const int* skip) {
    DPlan pl = plan(g, elementwise);
    if (!pl.ok || !encode_fn()) return -1;
    if ((long long)pl.bytes > MAX_PLANE_BYTES) {
        GemmArgs lo, hi;
        if (halve(g, lo, hi)) {
            const int a = launch_zgemm_digits(lo, elementwise, stream, workspace, workspace_bytes, skip);
            if (a < 0) return a;
            const int b = launch_zgemm_digits(hi, elementwise, stream, workspace, workspace_bytes, skip);
            return b < 0 ? b : a + b;
        }
    }
    if (!workspace || workspace_bytes < pl.bytes) return -2;
    DigitGemm& d = pl.d;
    uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
    auto side = [&](bool p) {
        const bool a = p != (d.swapped != 0);
        DigitSide s;
        std::memset(&s, 0, sizeof(s));
        if (a) {
            s.src = g.A; s.s_r = g.a_m; s.s_ki = g.a_ki; s.s_ko = g.a_ko; s.s_bi = g.a_bi; s.s_bo = g.a_bo;
            s.R = g.M; s.conj = g.conjA;
        } else {
            s.src = g.B; s.s_r = g.b_n; s.s_ki = g.b_ki; s.s_ko = g.b_ko; s.s_bi = g.b_bi; s.s_bo = g.b_bo;
            s.R = g.N; s.conj = g.conjB;
        }
        s.Ki = g.Ki;
        s.Ko = g.Ko;
        s.Bi = (p ? d.p_vbi : d.q_vbi) ? g.Bi : 1;
        s.Bo = (p ? d.p_vbo : d.q_vbo) ? g.Bo : 1;
        s.embed = p ? 0 : 1;
        s.Rpad = p ? d.Pp : d.Qp / 2;
        s.Kc = pl.Kp / 2;
        s.rows = p ? pl.np * d.Pp : pl.nq * d.Qp;
        s.planes = reinterpret_cast<uint16_t*>(ws + (p ? pl.p_off : pl.q_off));
        s.exps = reinterpret_cast<int*>(ws + (p ? pl.ep_off : pl.eq_off));
        if (elementwise) {
            s.mag = reinterpret_cast<uint16_t*>(ws + (p ? pl.mp_off : pl.mq_off));
            s.l1 = reinterpret_cast<unsigned long long*>(ws + (p ? pl.lp_off : pl.lq_off));
        }
        return s;
    };
    const DigitSide sp = side(true), sq = side(false);
    const int nbp = (int)((pl.np * d.Pp + PK_ROWS - 1) / PK_ROWS), nbq = (int)((pl.nq * (d.Qp / 2) + PK_ROWS - 1) / PK_ROWS);
    const int Kc = pl.Kp / 2;
    int launches = 0;
    // short K: one block per 32 rows finds the exponents and writes the
    // digits; long K: exponents first, K cut into blocks of 128
    const int one = Kc <= 256;
    const int kb = one ? Kc : 128;
    const dim3 grid(nbp + nbq, (Kc + kb - 1) / kb);
    if (!one) {
        if (cudaMemsetAsync(ws + pl.ep_off, 0, pl.p_off - pl.ep_off, stream) != cudaSuccess) return -1;
        launch(digit_max_kernel, grid, PK_THREADS, 0, stream, sp, sq, nbp, kb, skip);
        ++launches;
    }
    d.marked = elementwise ? reinterpret_cast<int*>(ws) + 1 : nullptr;
    launch(digit_pack_kernel, grid, PK_THREADS, 0, stream, sp, sq, nbp, kb, one, d.marked, skip);
    ++launches;
    CUtensorMap mP, mQ;
    if (!make_map3(&mP, sp.planes, sp.rows, pl.Kp, BM) || !make_map3(&mQ, sq.planes, sq.rows, pl.Kp, BN)) return -1;
    {
        static std::mutex mu;
        static bool set[64] = {};
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= 64) dev = 0;
        std::lock_guard<std::mutex> lock(mu);
        if (!set[dev]) {
            if (cudaFuncSetAttribute(digit_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES) !=
                cudaSuccess)
                return -1;
            set[dev] = true;
        }
    }
    d.expP = sp.exps;
    d.expQ = sq.exps;
    d.W = d.nsplit > 1 ? reinterpret_cast<cplx*>(ws + pl.w_off) : nullptr;
    d.err = reinterpret_cast<int*>(ws);
    d.skip = skip;
    d.stall_ns = test_take_tc_stall();
    if (elementwise) {
        d.mask = reinterpret_cast<uint32_t*>(ws + pl.mask_off);
        d.list = reinterpret_cast<uint32_t*>(ws + pl.list_off);
        d.magP = sp.mag;
        d.magQ = sq.mag;
        d.l1P = sp.l1;
        d.l1Q = sq.l1;
        const long long tiles = (long long)(d.Pp / 32) * d.n_qtiles * d.batches;
        if (d.Kc >= 8192 && tiles < 4 * N_SM) launch(digit_check_kernel<true>, (unsigned)tiles, CK_THREADS, 0, stream, d);
        else launch(digit_check_kernel<false>, (unsigned)((tiles + CK_WARPS - 1) / CK_WARPS), CK_THREADS, 0, stream, d);
        ++launches;
    }
    const long long nt = (long long)d.n_ptiles * d.n_qtiles * d.batches * d.nsplit;
    launch(digit_gemm_kernel, (unsigned)std::min<long long>(nt, N_SM), THREADS, SMEM_BYTES, stream, mP, mQ, d);
    ++launches;
    if (elementwise) {
        launch(digit_fix_kernel, N_SM, FX_THREADS, 0, stream, d);
        ++launches;
    }
    if (d.nsplit > 1) launches += launch_splitk_f64(g, d.nsplit, d.W, stream);
    return launches;
}
