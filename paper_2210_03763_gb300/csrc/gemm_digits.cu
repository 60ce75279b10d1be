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
// conversion to FP64.  Against the 53-bit products and sums of an FMA chain
// the error is smaller (measured, uniform operands, rms relative to |row|
// |column|: 7e-18 at K = 64, below the 3.3e-17 of an FMA chain).
//
// Why: GB300's FP64 pipe gives 1.06 TFLOP/s; 34 bf16 products give one FP64
// product at up to 1908 / 34 = 56 TFLOP/s.  Measured, packing included, against
// the FMA kernels: 128 x 16384 x 128 in batches of 16 28.1 -> 2.04 ms (16.8
// TFLOP/s), 128 x 128 x 16384 in batches of 16 40 -> 2.9 ms, 4096 x 64 x 64 in
// batches of 4 464 -> 64 us, 64 x 4096 x 256 463 -> 99 us (55 and 93 us since
// the MMAs are issued from a uniform warp).
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

// Row exponents over blocks of K (long K only): exps zeroed before.
__global__ void __launch_bounds__(PK_THREADS) digit_max_kernel(DigitSide sp, DigitSide sq, int nbp, int kb) {
    pdl_begin();
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
                                                               int one_pass) {
    pdl_begin();
    const bool isp = (int)blockIdx.x < nbp;
    const DigitSide& s = isp ? sp : sq;
    const long long f0 = (long long)(isp ? blockIdx.x : blockIdx.x - nbp) * PK_ROWS;
    __shared__ const cplx* base[PK_ROWS];
    __shared__ int mx[PK_ROWS];
    __shared__ cplx tile[PK_KT][PK_ROWS + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long nrow = (long long)s.Rpad * s.Bi * s.Bo;
    if (threadIdx.x < PK_ROWS) {
        base[threadIdx.x] = row_base(s, f0 + threadIdx.x);
        mx[threadIdx.x] = 0;
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
            if (f >= nrow || k >= s.Kc) continue;
            uint16_t* o = s.planes + (s.embed ? 2 * f : f) * 2LL * s.Kc + 2LL * k;
            if (!base[r] || mx[r] == 0x7FF) {   // padding; rows that the epilogue recomputes
#pragma unroll
                for (int q = 0; q < ND; ++q) {
                    *reinterpret_cast<uint32_t*>(o + q * plane) = 0u;
                    if (s.embed) *reinterpret_cast<uint32_t*>(o + q * plane + 2LL * s.Kc) = 0u;
                }
                continue;
            }
            const cplx v = tile[lane][r];
            const unsigned long long tr = biased_digits(v.x, mx[r]), ti = biased_digits(s.conj ? -v.y : v.y, mx[r]);
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
        }
        __syncthreads();
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
    cplx* W;                     // partial sums of split K (layout of splitk_f64_kernel)
    int* err;
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

// One output in plain FP64 (rows with infinities or NaNs), over this work
// item's K range.
__device__ __noinline__ cplx plain_output(const GemmArgs& g, int m, int n, int bi, int bo, int k0, int k1) {
    const cplx* A = g.A + bi * g.a_bi + bo * g.a_bo + m * g.a_m;
    const cplx* B = g.B + bi * g.b_bi + bo * g.b_bo + n * g.b_n;
    cplx s = make_double2(0.0, 0.0);
    for (int k = k0; k < k1; ++k) {
        cplx a = A[(k % g.Ki) * g.a_ki + (k / g.Ki) * g.a_ko], b = B[(k % g.Ki) * g.b_ki + (k / g.Ki) * g.b_ko];
        if (g.conjA) a.y = -a.y;
        if (g.conjB) b.y = -b.y;
        s.x = fma(a.x, b.x, s.x);
        s.x = fma(-a.y, b.y, s.x);
        s.y = fma(a.x, b.y, s.y);
        s.y = fma(a.y, b.x, s.y);
    }
    return s;
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
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mdone + 1);

    // an earlier launch on this workspace gave up: do nothing (the host
    // reports the error at its next check)
    __shared__ int s_skip;
    if (threadIdx.x == 0) s_skip = *(volatile int*)ea.err;
    __syncthreads();
    if (s_skip) return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nchunk = (ea.nst + CHUNK_ST - 1) / CHUNK_ST;
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
    // plane rows (complex P rows, real Q rows) where batch b starts
    auto row0 = [&](int b, int vbi, int vbo, int pad) {
        const int bi = b % ea.g.Bi, bo = b / ea.g.Bi;
        return ((vbi ? bi : 0) + (vbo ? bo * (vbi ? ea.g.Bi : 1) : 0)) * pad;
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
                const int prow = row0(b, ea.p_vbi, ea.p_vbo, ea.Pp) + pt * BM;
                const int qrow = row0(b, ea.q_vbi, ea.q_vbo, ea.Qp) + qt * BN;
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
        const bool a1 = ea.g.alpha.x == 1.0 && ea.g.alpha.y == 0.0;
        const bool b0 = ea.g.beta.x == 0.0 && ea.g.beta.y == 0.0;
        const bool b1 = ea.g.beta.x == 1.0 && ea.g.beta.y == 0.0;
        unsigned cg = 0;
        bool ok = true;
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
            if (p >= ea.Pn) continue;
            const int bi = b % ea.g.Bi, bo = b / ea.g.Bi;
            const int ep = ea.expP[row0(b, ea.p_vbi, ea.p_vbo, ea.Pp) + p];
            const int* eq = ea.expQ + row0(b, ea.q_vbi, ea.q_vbo, ea.Qp) / 2;
#pragma unroll
            for (int j = 0; j < DCOLS; j += 2) {
                const int q = (qt * BN + col0 + j) >> 1;
                if (q >= ea.Qn) continue;
                const int e = eq[q];
                const int m = ea.swapped ? q : p, n = ea.swapped ? p : q;
                cplx r;
                if (ep == 0x7FF || e == 0x7FF) {
                    r = plain_output(ea.g, m, n, bi, bo, st0 * BK / 2, min(ea.g.Ki * ea.g.Ko, st1 * BK / 2));
                } else {
                    const int sc = max(ep, 1) + max(e, 1) - 2 * 1022 - 70;   // E_p + E_q - 110 + 40
                    r = make_double2(to_double(sh[j], sl[j], sc), to_double(sh[j + 1], sl[j + 1], sc));
                }
                if (ea.nsplit > 1) {
                    ea.W[(((long long)ks * ea.batches + b) * ea.g.N + n) * ea.g.M + m] = r;
                    continue;
                }
                cplx* cp = ea.g.C + bi * ea.g.c_bi + bo * ea.g.c_bo + m * ea.g.c_m + n * ea.g.c_n;
                if (!a1) {
                    const cplx v = r;
                    r.x = ea.g.alpha.x * v.x - ea.g.alpha.y * v.y;
                    r.y = ea.g.alpha.x * v.y + ea.g.alpha.y * v.x;
                }
                if (!b0) {
                    const cplx o = *cp;
                    if (b1) {
                        r.x += o.x;
                        r.y += o.y;
                    } else {
                        r.x += ea.g.beta.x * o.x - ea.g.beta.y * o.y;
                        r.y += ea.g.beta.x * o.y + ea.g.beta.y * o.x;
                    }
                }
                *cp = r;
            }
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
    size_t p_off = 0, q_off = 0, ep_off = 0, eq_off = 0, w_off = 0, bytes = 0;
};

DPlan plan(const GemmArgs& g) {
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
    pl.p_off = take((size_t)ND * pl.np * d.Pp * pl.Kp * 2);
    pl.q_off = take((size_t)ND * pl.nq * d.Qp * pl.Kp * 2);
    if (d.nsplit > 1) pl.w_off = take((size_t)d.nsplit * d.batches * g.M * (size_t)g.N * sizeof(cplx));
    pl.bytes = off;
    pl.ok = pl.np * d.Pp < (1LL << 31) && pl.nq * d.Qp < (1LL << 31);
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
// of packing both sides plus the tile work (measured at the border: 4096 x 64 x
// 64 280 us on the FP64 pipe, 48 in digits; 64 x 64 x 64 9 us and 13).
bool digits_wanted(const GemmArgs& g) {
    const double K = (double)g.Ki * g.Ko, macs = (double)g.M * g.N * K * g.Bi * (double)g.Bo;
    if (std::min(g.M, g.N) < 16 || std::max(g.M, g.N) < 32 || K < 16) return false;
    DPlan pl = plan(g);
    if (!pl.ok || !encode_fn()) return false;
    const double f64_us = 4.0 + 8.0 * macs / 1.0e6;
    const double chunks = (double)pl.d.n_ptiles * pl.d.n_qtiles * pl.d.batches * ((pl.d.nst + CHUNK_ST - 1) / CHUNK_ST);
    const double us = 16.0 + 6.5 * std::max(1.0, chunks / N_SM) + (double)pl.bytes / 2.0e6;
    return us < f64_us;
}

size_t digits_workspace_bytes(const GemmArgs& g) {
    DPlan pl = plan(g);
    if (!pl.ok) return 0;
    if ((long long)pl.bytes > MAX_PLANE_BYTES) {
        GemmArgs lo, hi;
        if (halve(g, lo, hi)) return std::max(digits_workspace_bytes(lo), digits_workspace_bytes(hi));
    }
    return pl.bytes;
}

int launch_zgemm_digits(const GemmArgs& g, cudaStream_t stream, void* workspace, size_t workspace_bytes) {
    DPlan pl = plan(g);
    if (!pl.ok || !encode_fn()) return -1;
    if ((long long)pl.bytes > MAX_PLANE_BYTES) {
        GemmArgs lo, hi;
        if (halve(g, lo, hi)) {
            const int a = launch_zgemm_digits(lo, stream, workspace, workspace_bytes);
            if (a < 0) return a;
            const int b = launch_zgemm_digits(hi, stream, workspace, workspace_bytes);
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
        launch(digit_max_kernel, grid, PK_THREADS, 0, stream, sp, sq, nbp, kb);
        ++launches;
    }
    launch(digit_pack_kernel, grid, PK_THREADS, 0, stream, sp, sq, nbp, kb, one);
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
    const long long nt = (long long)d.n_ptiles * d.n_qtiles * d.batches * d.nsplit;
    launch(digit_gemm_kernel, (unsigned)std::min<long long>(nt, N_SM), THREADS, SMEM_BYTES, stream, mP, mQ, d);
    ++launches;
    if (d.nsplit > 1) launches += launch_splitk_f64(g, d.nsplit, d.W, stream);
    return launches;
}
