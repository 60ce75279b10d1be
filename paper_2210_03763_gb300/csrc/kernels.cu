// Vector, reduction and small-matrix kernels of the TDVP update.
//
// Each of G blocks of a reduction writes a partial sum for a contiguous chunk
// of the vector, and every consumer sums the G partials in the same fixed order,
// so repeated runs are bitwise identical and every block of a kernel sees the
// same reduced value.  Atomics only count the blocks that have finished.
#include "common.cuh"
#include <cooperative_groups.h>
#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>
#include <sched.h>

namespace {

constexpr int T = RED_THREADS;

__device__ __forceinline__ cplx cadd(cplx a, cplx b) { return make_double2(a.x + b.x, a.y + b.y); }
// The vector kernels below are bound by GB300's FP64 pipe (about 1/64 of its
// FP32 rate), not by HBM, so the complex multiply-accumulates are written as
// four fused multiply-adds (s += conj(a) b, x -= a h) instead of two
// multiplies, two fused operations and two adds.
__device__ __forceinline__ void acc_cdotc(cplx& s, cplx a, cplx b) {
    s.x = fma(a.x, b.x, s.x);
    s.x = fma(a.y, b.y, s.x);
    s.y = fma(a.x, b.y, s.y);
    s.y = fma(-a.y, b.x, s.y);
}
__device__ __forceinline__ void sub_cmul(cplx& x, cplx a, cplx h) {
    x.x = fma(-a.x, h.x, x.x);
    x.x = fma(a.y, h.y, x.x);
    x.y = fma(-a.x, h.y, x.y);
    x.y = fma(-a.y, h.x, x.y);
}
__device__ __forceinline__ void acc_cmul(cplx& x, cplx a, cplx h) {
    x.x = fma(a.x, h.x, x.x);
    x.x = fma(-a.y, h.y, x.x);
    x.y = fma(a.x, h.y, x.y);
    x.y = fma(a.y, h.x, x.y);
}

__device__ __forceinline__ void chunk_of(long long n, int G, long long& lo, long long& hi) {
    long long c = (n + G - 1) / G;
    lo = (long long)blockIdx.x * c;
    hi = lo + c < n ? lo + c : n;
}

__device__ double block_sum_d(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
    return r;
}

// Sum the G partials of nv projections (partial[i*G + g]) into sh_h[0..nv):
// one warp per projection (a serial sum of 304 partials took 4 us in every
// block of every launch), lanes in fixed order.
__device__ __forceinline__ cplx warp_sum_c(cplx v) {
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}
__device__ void reduce_partials_to_shared(const cplx* partial, int nv, int G, cplx* sh_h) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < nv; i += blockDim.x >> 5) {
        cplx s = make_double2(0.0, 0.0);
        for (int g = lane; g < G; g += 32) s = cadd(s, partial[(long long)i * G + g]);
        s = warp_sum_c(s);
        if (lane == 0) sh_h[i] = s;
    }
    __syncthreads();
}

// By one warp; the sum in every lane.
__device__ double reduce_norm_partials(const double* partial, int G) {
    double s = 0.0;
    for (int g = threadIdx.x & 31; g < G; g += 32) s += partial[g];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// ---------------------------------------------------------------- kernels
// conj(V_i) . w over [lo, hi) for C consecutive vectors, summed over the warp
// (in every lane).
template <int C>
__device__ __forceinline__ void warp_dots(const cplx* V, long long ld, const cplx* w, long long lo, long long hi,
                                          int first, int stride, cplx* s) {
#pragma unroll
    for (int c = 0; c < C; ++c) s[c] = make_double2(0.0, 0.0);
    for (long long e = lo + first; e < hi; e += stride) {
        const cplx x = w[e];
#pragma unroll
        for (int c = 0; c < C; ++c) acc_cdotc(s[c], V[c * ld + e], x);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) s[c] = warp_sum_c(s[c]);
}

// Partial dots conj(V_i) . w, i < nv, over this block's chunk into
// partial[i*G + block].  Long chunks: every warp takes a slice of the chunk,
// four vectors at a time (w is read once per four); short chunks: one vector
// per warp, so that no sum crosses warps.
constexpr int SHORT_CHUNK = 256;
struct DotSmem {
    cplx w[T / 32][KRYLOV_MMAX + 1];
};
__device__ void block_dots(const cplx* V, long long ld, int nv, const cplx* w, long long lo, long long hi, int G,
                           cplx* partial, DotSmem& sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cplx s[4];
    if (hi - lo <= SHORT_CHUNK) {
        for (int i = warp; i < nv; i += T / 32) {
            warp_dots<1>(V + (long long)i * ld, ld, w, lo, hi, lane, 32, s);
            if (lane == 0) partial[(long long)i * G + blockIdx.x] = s[0];
        }
        return;
    }
    for (int i = 0; i < nv; i += 4) {
        const cplx* v = V + (long long)i * ld;
        const int c = nv - i < 4 ? nv - i : 4;
        if (c == 4) warp_dots<4>(v, ld, w, lo, hi, threadIdx.x, T, s);
        else if (c == 3) warp_dots<3>(v, ld, w, lo, hi, threadIdx.x, T, s);
        else if (c == 2) warp_dots<2>(v, ld, w, lo, hi, threadIdx.x, T, s);
        else warp_dots<1>(v, ld, w, lo, hi, threadIdx.x, T, s);
        if (lane == 0)
            for (int q = 0; q < c; ++q) sm.w[warp][i + q] = s[q];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nv; i += T) {
        cplx a = sm.w[0][i];
        for (int q = 1; q < T / 32; ++q) a = cadd(a, sm.w[q][i]);
        partial[(long long)i * G + blockIdx.x] = a;
    }
}

__global__ void __launch_bounds__(T) dots_kernel(const cplx* V, long long ld, int nv, const cplx* w, long long n, int G,
                                                 cplx* partial) {
    pdl_begin();
    __shared__ DotSmem sm;
    long long lo, hi;
    chunk_of(n, G, lo, hi);
    block_dots(V, ld, nv, w, lo, hi, G, partial, sm);
}

// First pass of Arnoldi: h = sum of the partials of all nv projections
// (stored to h_out), w -= sum_i V_i h_i, partial dots of the new w.
__global__ void __launch_bounds__(T) orth_first_kernel(const cplx* V, long long ld, int nv, const cplx* partial_in,
                                                       cplx* w, long long n, int G, cplx* partial_dots, cplx* h_out) {
    pdl_begin();
    __shared__ cplx sh_h[KRYLOV_MMAX + 1];
    __shared__ DotSmem sm;
    reduce_partials_to_shared(partial_in, nv, G, sh_h);
    if (blockIdx.x == 0 && threadIdx.x < nv) h_out[threadIdx.x] = sh_h[threadIdx.x];
    long long lo, hi;
    chunk_of(n, G, lo, hi);
    for (long long e = lo + threadIdx.x; e < hi; e += T) {
        cplx x = w[e];
        for (int i = 0; i < nv; ++i) sub_cmul(x, V[(long long)i * ld + e], sh_h[i]);
        w[e] = x;
    }
    __syncthreads();
    block_dots(V, ld, nv, w, lo, hi, G, partial_dots, sm);
}

// First pass of Lanczos.  H is Hermitian (up to the rounding of its
// contractions), so only v_j and v_{j-1} have components in w beyond
// rounding: w -= v_j h + v_{j-1} beta_{j-1} with h = v_j^H w, then the
// partial dots of the new w with the whole basis, whose second pass removes
// what is left.  Two sweeps over the basis instead of four: the vector work
// is bound by the FP64 pipe.
__global__ void __launch_bounds__(T) lanczos_first_kernel(const cplx* V, long long ld, int j, const cplx* partial_in,
                                                          const KrylovScalars* ks, cplx* w, long long n, int G,
                                                          cplx* partial_dots, cplx* h_out) {
    pdl_begin();
    __shared__ cplx sh_h[1];
    __shared__ DotSmem sm;
    reduce_partials_to_shared(partial_in, 1, G, sh_h);
    const cplx h = sh_h[0];
    const double b = j > 0 ? ks->beta[j - 1] : 0.0;
    if (blockIdx.x == 0 && threadIdx.x <= j) h_out[threadIdx.x] = threadIdx.x == j ? h : make_double2(0.0, 0.0);
    long long lo, hi;
    chunk_of(n, G, lo, hi);
    const cplx* vj = V + (long long)j * ld;
    for (long long e = lo + threadIdx.x; e < hi; e += T) {
        cplx x = w[e];
        sub_cmul(x, vj[e], h);
        if (j > 0) {
            const cplx v = vj[e - ld];
            x.x = fma(-b, v.x, x.x);
            x.y = fma(-b, v.y, x.y);
        }
        w[e] = x;
    }
    __syncthreads();
    block_dots(V, ld, j + 1, w, lo, hi, G, partial_dots, sm);
}

__device__ void krylov_scalars_step(KrylovScalars* ks, const cplx* h1, const cplx* h2, const double* beta_partial,
                                    int G, int j, double zr, double zi, double tol, int arnoldi, const Publish& pub);

// The fields are written; make them visible to the host, then the number.
__device__ __forceinline__ void publish(const Publish& pub) {
    if (pub.tc_flag && *(volatile const int*)pub.tc_flag) pub.hs->tc_flag = 1;
    __threadfence_system();
    *(volatile unsigned*)&pub.hs->seq = pub.seq;
}

// Second pass: h = sum of the partials, w -= sum_i V_i h_i, |w|^2.  The last
// block to finish turns the sums into the step's scalars (alpha, beta, the
// exponential of the projected matrix, the error estimate).
__global__ void __launch_bounds__(T) orth_second_kernel(const cplx* V, long long ld, int nv, const cplx* partial_in,
                                                        cplx* w, long long n, int G, double* partial_norm,
                                                        KrylovScalars* ks, const cplx* h1, double zr, double zi,
                                                        double tol, int arnoldi, Publish pub) {
    pdl_begin();
    __shared__ cplx sh_h[KRYLOV_MMAX + 1];
    __shared__ double shd[T / 32];
    __shared__ int last;
    reduce_partials_to_shared(partial_in, nv, G, sh_h);
    long long lo, hi;
    chunk_of(n, G, lo, hi);
    double s = 0.0;
    for (long long e = lo + threadIdx.x; e < hi; e += T) {
        cplx x = w[e];
        for (int i = 0; i < nv; ++i) sub_cmul(x, V[(long long)i * ld + e], sh_h[i]);
        w[e] = x;
        s = fma(x.x, x.x, fma(x.y, x.y, s));
    }
    s = block_sum_d(s, shd);
    if (threadIdx.x == 0) {
        partial_norm[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(&ks->arrived, 1u) == gridDim.x - 1;
        if (last) ks->arrived = 0u;
        __threadfence();
    }
    __syncthreads();
    if (last && threadIdx.x < 32) krylov_scalars_step(ks, h1, sh_h, partial_norm, G, nv - 1, zr, zi, tol, arnoldi, pub);
}

__global__ void norm2_partial_kernel(const cplx* x, long long n, int G, double* partial) {
    pdl_begin();
    __shared__ double shd[T / 32];
    long long lo, hi;
    chunk_of(n, G, lo, hi);
    double s = 0.0;
    for (long long e = lo + threadIdx.x; e < hi; e += blockDim.x) s += x[e].x * x[e].x + x[e].y * x[e].y;
    s = block_sum_d(s, shd);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void scale_copy_kernel(const cplx* x, long long n, const double* scale, cplx* y) {
    pdl_begin();
    double f = scale[0];
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        cplx v = x[e];
        y[e] = make_double2(v.x * f, v.y * f);
    }
}

// x <- x * sqrt(sum(pr) / sum(px)): rescale x to the norm given by the
// partial sums pr (each block sums both partial lists in the same order).
__global__ void rescale_to_norm_kernel(cplx* x, long long n, const double* px, int Gx, const double* pr, int Gr) {
    pdl_begin();
    __shared__ double f;
    if (threadIdx.x < 32) {
        const double a = reduce_norm_partials(px, Gx), b = reduce_norm_partials(pr, Gr);
        if (threadIdx.x == 0) f = a > 0.0 ? sqrt(b / a) : 1.0;
    }
    __syncthreads();
    const double ff = f;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        cplx v = x[e];
        x[e] = make_double2(v.x * ff, v.y * ff);
    }
}

__global__ void combine_kernel(const cplx* V, long long ld, int nv, const KrylovScalars* ks, cplx* y,
                               long long n) {
    pdl_begin();
    __shared__ cplx c[KRYLOV_MMAX];
    if (threadIdx.x < nv) {
        cplx ci = ks->c[nv - 1][threadIdx.x];
        c[threadIdx.x] = make_double2(ci.x * ks->nrm0, ci.y * ks->nrm0);
    }
    __syncthreads();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        cplx s = make_double2(0.0, 0.0);
        for (int i = 0; i < nv; ++i) acc_cmul(s, V[(long long)i * ld + e], c[i]);
        y[e] = s;
    }
}

// 1/k for the Taylor terms.
__constant__ double INV_K[41] = {0.0,      1.0 / 1,  1.0 / 2,  1.0 / 3,  1.0 / 4,  1.0 / 5,  1.0 / 6,  1.0 / 7,  1.0 / 8,
                                 1.0 / 9,  1.0 / 10, 1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16, 1.0 / 17,
                                 1.0 / 18, 1.0 / 19, 1.0 / 20, 1.0 / 21, 1.0 / 22, 1.0 / 23, 1.0 / 24, 1.0 / 25, 1.0 / 26,
                                 1.0 / 27, 1.0 / 28, 1.0 / 29, 1.0 / 30, 1.0 / 31, 1.0 / 32, 1.0 / 33, 1.0 / 34, 1.0 / 35,
                                 1.0 / 36, 1.0 / 37, 1.0 / 38, 1.0 / 39, 1.0 / 40};

// High words of |re|, |im|: ordered like the magnitudes, compared without the
// FP64 pipe.
__device__ __forceinline__ unsigned mag_hi(cplx v) {
    const unsigned a = (unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, b = (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu;
    return a > b ? a : b;
}
// Every lane's term is below 2^-60 of the largest sum: the series is done.
__device__ __forceinline__ bool series_done(cplx term, cplx sum) {
    const unsigned tm = __reduce_max_sync(0xffffffffu, mag_hi(term)), sm = __reduce_max_sync(0xffffffffu, mag_hi(sum));
    return (unsigned long long)tm + (60u << 20) <= sm || tm == 0u;
}

// Sub-steps that keep |z| norm / n_sub <= 1/2: bounded also for non-finite or
// absurd norms (a NaN state is reported through the nonfinite flag, never by
// a runaway loop).
__device__ __forceinline__ int taylor_substeps(double want) {
    return (want >= 1.0 && want < 65536.0) ? (int)ceil(want) : (want >= 65536.0 ? 65536 : 1);
}

// exp(z T) e_1 for the real symmetric tridiagonal T (diag a[0..m), off-diag
// b[0..m-1)), m <= 32, by the truncated Taylor series of the matrix
// exponential applied to the vector, with the step z split into n_sub equal
// substeps so that |z/n_sub| * ||T||_inf <= 1/2 (the "Taylor series" method of
// Moler & Van Loan, "Nineteen dubious ways to compute the exponential of a
// matrix", with scaling).  One warp; lane i holds component i.  The warp runs
// alone, so a term costs its FP64 instructions one after another: z is i or
// real in every caller but the general case, 1/k comes from a table and the
// stopping test is integer.
__device__ void tridiag_expm_warp(const double* a, const double* b, int m, double zr, double zi,
                                  cplx* out) {
    const int l = threadIdx.x & 31;
    const double ai = l < m ? a[l] : 0.0;
    const double bl = (l < m - 1) ? b[l] : 0.0;          // T(l, l+1)
    const double bu = (l >= 1 && l < m) ? b[l - 1] : 0.0; // T(l, l-1)
    double rs = fabs(ai) + fabs(bl) + fabs(bu);
    for (int o = 16; o > 0; o >>= 1) rs = fmax(rs, __shfl_xor_sync(0xffffffffu, rs, o));
    const int nsub = taylor_substeps(sqrt(zr * zr + zi * zi) * rs / 0.5);
    const double hr = zr / nsub, hi = zi / nsub;
    cplx u = make_double2(l == 0 ? 1.0 : 0.0, 0.0);
    for (int s = 0; s < nsub; ++s) {
        cplx term = u, sum = u;
        for (int k = 1; k <= 40; ++k) {
            // t = T term (lanes outside [0, m) have zero rows)
            const double xm_r = __shfl_up_sync(0xffffffffu, term.x, 1);
            const double xm_i = __shfl_up_sync(0xffffffffu, term.y, 1);
            const double xp_r = __shfl_down_sync(0xffffffffu, term.x, 1);
            const double xp_i = __shfl_down_sync(0xffffffffu, term.y, 1);
            const double tr = fma(bl, xp_r, fma(bu, xm_r, ai * term.x));
            const double ti = fma(bl, xp_i, fma(bu, xm_i, ai * term.y));
            // term = (h * t) / k
            if (hr == 0.0) {
                const double c = hi * INV_K[k];
                term = make_double2(-c * ti, c * tr);
            } else {
                term = make_double2((hr * tr - hi * ti) * INV_K[k], (hr * ti + hi * tr) * INV_K[k]);
            }
            sum = cadd(sum, term);
            if (series_done(term, sum)) break;
        }
        u = sum;
    }
    if (l < m) out[l] = u;
}

// |x|^2; the last block to finish sets the start scalars.
__global__ void __launch_bounds__(T) krylov_start_kernel(KrylovScalars* ks, const cplx* x, long long n, int G,
                                                         double* partial, unsigned* arrived) {
    pdl_begin();
    __shared__ double shd[T / 32];
    __shared__ int last;
    long long lo, hi;
    chunk_of(n, G, lo, hi);
    double s = 0.0;
    for (long long e = lo + threadIdx.x; e < hi; e += T) s = fma(x[e].x, x[e].x, fma(x[e].y, x[e].y, s));
    s = block_sum_d(s, shd);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(arrived, 1u) == gridDim.x - 1;
        if (last) *arrived = 0u;
        __threadfence();
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    double t = 0.0;
    for (int g = threadIdx.x; g < G; g += 32) t += __ldcg(partial + g);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) {
        const double n0 = sqrt(t);
        ks->nrm0 = n0;
        ks->inv_scale = n0 > 0.0 ? 1.0 / n0 : 0.0;
        ks->nonfinite = isfinite(n0) ? 0 : 1;
    }
}

// exp(z H) e_1 for the m x m matrix H, H(i, k) at Hs[32 k + i] in shared
// memory, m <= 31, by the scaled Taylor series as in tridiag_expm_warp:
// substeps with |z/n_sub| * ||H||_inf <= 1/2.  One warp; lane i holds
// component i; the vector goes round through `vec` (32 entries of shared
// memory).
__device__ void hess_expm_warp(const cplx* Hs, cplx* vec, int m, double zr, double zi, cplx* out) {
    const int l = threadIdx.x & 31;
    double rs = 0.0;
    if (l < m)
        for (int k = 0; k < m; ++k) {
            const cplx v = Hs[32 * k + l];
            rs += sqrt(v.x * v.x + v.y * v.y);
        }
    for (int o = 16; o > 0; o >>= 1) rs = fmax(rs, __shfl_xor_sync(0xffffffffu, rs, o));
    const int nsub = taylor_substeps(sqrt(zr * zr + zi * zi) * rs / 0.5);
    const double hr = zr / nsub, hi = zi / nsub;
    cplx u = make_double2(l == 0 ? 1.0 : 0.0, 0.0);
    for (int s = 0; s < nsub; ++s) {
        cplx term = u, sum = u;
        for (int k = 1; k <= 40; ++k) {
            __syncwarp();
            vec[l] = term;
            __syncwarp();
            cplx t = make_double2(0.0, 0.0);
            if (l < m) {
                // row l of the Hessenberg matrix starts at column l - 1
                for (int q = l > 0 ? l - 1 : 0; q < m; ++q) acc_cmul(t, Hs[32 * q + l], vec[q]);
            }
            const double inv = INV_K[k];
            term = make_double2((hr * t.x - hi * t.y) * inv, (hr * t.y + hi * t.x) * inv);
            sum = cadd(sum, term);
            if (series_done(term, sum)) break;
        }
        u = sum;
    }
    __syncwarp();
    if (l < m) out[l] = u;
}

// Scalars of step j by one warp: alpha_j, beta_j (Arnoldi: column j of the
// Hessenberg matrix), c = exp(z T) e_1, the error estimate and the status.
__device__ void krylov_scalars_step(KrylovScalars* ks, const cplx* h1, const cplx* h2, const double* beta_partial,
                                    int G, int j, double zr, double zi, double tol, int arnoldi, const Publish& pub) {
    __shared__ double a[32], b[32];
    __shared__ cplx hs[KRYLOV_MMAX * 32], vec[32];
    const int l = threadIdx.x & 31;
    double s = 0.0;
    for (int g = l; g < G; g += 32) s += __ldcg(beta_partial + g);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double bj = sqrt(s);
    bool bad;
    if (arnoldi) {
        // the whole column j: projections, the subdiagonal beta_j, zeros below
        const cplx col = l <= j ? cadd(h1[l], h2[l]) : make_double2(l == j + 1 ? bj : 0.0, 0.0);
        ks->hess[j][l] = col;
        for (int q = 0; q < j; ++q) hs[32 * q + l] = ks->hess[q][l];
        hs[32 * j + l] = col;
        __syncwarp();
        const cplx d = hs[33 * j];
        bad = !isfinite(d.x) || !isfinite(d.y);
        if (l == 0) {
            ks->beta[j] = bj;
            ks->alpha[j] = d.x;
        }
        hess_expm_warp(hs, vec, j + 1, zr, zi, ks->c[j]);
    } else {
        const double al = h1[j].x + h2[j].x;
        bad = !isfinite(al);
        a[l] = l < j ? ks->alpha[l] : l == j ? al : 0.0;
        b[l] = l < j ? ks->beta[l] : 0.0;
        __syncwarp();
        if (l == 0) {
            ks->alpha[j] = al;
            ks->beta[j] = bj;
        }
        tridiag_expm_warp(a, b, j + 1, zr, zi, ks->c[j]);
    }
    __syncwarp();
    if (l == 0) {
        const cplx cj = ks->c[j][j];
        const double err = bj * sqrt(cj.x * cj.x + cj.y * cj.y);
        ks->inv_scale = bj > 0.0 ? 1.0 / bj : 0.0;
        if (!isfinite(err) || bad) ks->nonfinite = 1;
        KrylovStatus& st = pub.hs->krylov[j];
        st.err = err;
        st.converged = (err <= tol) ? 1 : 0;
        st.nonfinite = ks->nonfinite;
        publish(pub);
    }
}

// ------------------------------------------------------------- small nodes
// The whole Krylov exponential x <- exp(z H) x of a node or link with s <= 96
// entries in one launch of one cluster: H_eff as a dense matrix (block terms
// hb_u, D_u x D_u or nullptr, and channel pairs sum_i Na_i (leg a) (x) G_i
// (leg b)), Lanczos (or Arnoldi when `arnoldi`) with the same passes,
// exponential and stopping rule as the multi-kernel path.  Status goes to ks.
//
// One SM's FP64 pipe (19 clk per warp-wide FMA) is the bound: an 81 x 81
// matvec alone is 7 us on it.  So the rows are split over the 8 SMs of a
// cluster; every CTA keeps the whole basis, computes its rows of w and its
// partial dots, and writes them into all CTAs' shared memory (three cluster
// barriers per iteration).  All CTAs sum the same partials in the same order,
// so they take the same decisions.  Warp 0 takes the projected exponential
// while the other warps already multiply the next vector.
// Measured: 225 us per run of a 2x2 step (one block on one SM) -> 54 us.
constexpr int SK_CL = 8;                                  // CTAs per cluster
constexpr int SK_THREADS = 256;
constexpr int SK_ROWS = (SMALL_S + SK_CL - 1) / SK_CL;    // rows per CTA (12), at most 16 for the group sums
static_assert(SK_ROWS <= 16, "16-lane groups");

struct SkSmem {
    cplx xa[SK_CL][32], xb[SK_CL][32];   // partial dots of every CTA, first and second pass
    double xn[SK_CL];                    // partial norms
    cplx xw[SMALL_S];                    // w, rows from every CTA
    cplx h1[32], h2[32], c[32], w[SK_ROWS];
    double alpha[32], beta[32];
    cplx hess[KRYLOV_MMAX * 32], hvec[32];   // Arnoldi: H(i, j) at [32 j + i]
    int done, conv, nonfin;
    double err;
};

__device__ __forceinline__ cplx group16_sum(cplx v) {
    for (int o = 8; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

__device__ cplx small_heff(int xr, int yc, int d0, int d1, int d2, const cplx* hb0, const cplx* hb1, const cplx* hb2,
                           const SmallPairs& pp) {
    const int x[3] = {xr % d0, (xr / d0) % d1, xr / (d0 * d1)};
    const int y[3] = {yc % d0, (yc / d0) % d1, yc / (d0 * d1)};
    const int dd[3] = {d0, d1, d2};
    const cplx* hb[3] = {hb0, hb1, hb2};
    cplx h = make_double2(0.0, 0.0);
    for (int u = 0; u < 3; ++u) {
        if (!hb[u]) continue;
        bool diag = true;
        for (int v = 0; v < 3; ++v)
            if (v != u && x[v] != y[v]) diag = false;
        if (diag) h = cadd(h, hb[u][x[u] + dd[u] * y[u]]);
    }
    for (int p = 0; p < pp.np; ++p) {
        const int a = pp.a[p], b = pp.b[p], w = 3 - a - b;
        if (x[w] != y[w]) continue;
        const long long Da2 = (long long)dd[a] * dd[a], Db2 = (long long)dd[b] * dd[b];
        const long long ia = x[a] + (long long)dd[a] * y[a], ib = x[b] + (long long)dd[b] * y[b];
        for (int i = 0; i < pp.r[p]; ++i) acc_cmul(h, pp.Na[p][i * Da2 + ia], pp.G[p][i * Db2 + ib]);
    }
    return h;
}

__global__ void __cluster_dims__(SK_CL, 1, 1) __launch_bounds__(SK_THREADS)
    small_krylov_kernel(int d0, int d1, int d2, const cplx* hb0, const cplx* hb1, const cplx* hb2, SmallPairs pp,
                        cplx* x, double zr, double zi, double tol, int mmax, int arnoldi, Publish pub) {
    pdl_begin();
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ cplx smem_c[];
    __shared__ SkSmem sm;
    const int s = d0 * d1 * d2, R = (s + SK_CL - 1) / SK_CL;
    const int rank = (int)cl.block_rank(), r0 = rank * R, nr = max(0, min(R, s - r0));
    cplx* Hs = smem_c;              // own rows: H(r0 + r, k) at [k * R + r]
    cplx* V = Hs + R * s;           // (mmax + 1) * s
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g16 = tid >> 4, l16 = tid & 15;
    for (int e = tid; e < nr * s; e += SK_THREADS) {
        const int r = e % nr, k = e / nr;
        Hs[k * R + r] = small_heff(r0 + r, k, d0, d1, d2, hb0, hb1, hb2, pp);
    }
    for (int e = tid; e < s; e += SK_THREADS) V[e] = x[e];
    __syncthreads();
    double nrm0 = 0.0;
    for (int e = lane; e < s; e += 32) nrm0 = fma(V[e].x, V[e].x, fma(V[e].y, V[e].y, nrm0));
    for (int o = 16; o > 0; o >>= 1) nrm0 += __shfl_xor_sync(0xffffffffu, nrm0, o);
    nrm0 = sqrt(nrm0);
    cl.sync();                      // every CTA has read x; all are running (remote writes may start)
    if (nrm0 == 0.0 || !isfinite(nrm0)) {
        if (rank == 0 && tid == 0) {
            KrylovStatus& st = pub.hs->krylov[0];
            st.err = 0.0;
            st.converged = nrm0 == 0.0;
            st.nonfinite = nrm0 != 0.0;
            st.iters = 0;
            publish(pub);
        }
        return;
    }
    if (tid == 0) sm.nonfin = 0;
    const double inv0 = 1.0 / nrm0;
    for (int e = tid; e < s; e += SK_THREADS) V[e] = make_double2(V[e].x * inv0, V[e].y * inv0);
    __syncthreads();
    // own rows of w = H v, 16 lanes per row, by `nt` threads numbered from t
    auto matvec = [&](const cplx* v, int t, int nt) {
        for (int q = t; q < ((nr * 16 + 31) & ~31); q += nt) {
            const int r = q >> 4;
            cplx a = make_double2(0.0, 0.0);
            if (r < nr)
                for (int k = q & 15; k < s; k += 16) acc_cmul(a, Hs[k * R + r], v[k]);
            a = group16_sum(a);
            if (r < nr && (q & 15) == 0) sm.w[r] = a;
        }
    };
    // partial dots of own rows with v_i, i0 <= i < i1, into every CTA's buf
    auto dots = [&](int i0, int i1, cplx(*buf)[32]) {
        const int n = i1 - i0;
        for (int q = g16; q < ((n + 1) & ~1); q += SK_THREADS / 16) {   // both groups of a warp stay together
            cplx d = make_double2(0.0, 0.0);
            if (q < n && l16 < nr) acc_cdotc(d, V[(i0 + q) * s + r0 + l16], sm.w[l16]);
            d = group16_sum(d);
            if (q < n && l16 < SK_CL) cl.map_shared_rank(&buf[rank][0], l16)[q] = d;
        }
    };
    matvec(V, tid, SK_THREADS);
    int j = 0;
    for (;; ++j) {
        __syncthreads();
        const int first = arnoldi ? 0 : j;   // first pass: all vectors, or v_j and beta v_{j-1}
        dots(first, j + 1, sm.xa);
        cl.sync();
        if (tid <= j) {
            cplx h = make_double2(0.0, 0.0);
            if (tid >= first)
                for (int q = 0; q < SK_CL; ++q) h = cadd(h, sm.xa[q][tid - first]);
            sm.h1[tid] = h;
        }
        __syncthreads();
        if (tid < nr) {
            cplx w = sm.w[tid];
            for (int i = first; i <= j; ++i) sub_cmul(w, V[i * s + r0 + tid], sm.h1[i]);
            if (!arnoldi && j > 0) {
                const cplx v = V[(j - 1) * s + r0 + tid];
                w.x = fma(-sm.beta[j - 1], v.x, w.x);
                w.y = fma(-sm.beta[j - 1], v.y, w.y);
            }
            sm.w[tid] = w;
        }
        __syncthreads();
        dots(0, j + 1, sm.xb);
        cl.sync();
        if (tid <= j) {
            cplx h = make_double2(0.0, 0.0);
            for (int q = 0; q < SK_CL; ++q) h = cadd(h, sm.xb[q][tid]);
            sm.h2[tid] = h;
        }
        __syncthreads();
        if (warp == 0) {
            cplx w = make_double2(0.0, 0.0);
            double n2 = 0.0;
            if (lane < nr) {
                w = sm.w[lane];
                for (int i = 0; i <= j; ++i) sub_cmul(w, V[i * s + r0 + lane], sm.h2[i]);
                n2 = fma(w.x, w.x, w.y * w.y);
            }
            for (int o = 8; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
            n2 = __shfl_sync(0xffffffffu, n2, 0);
            for (int q = 0; q < SK_CL; ++q) {
                if (lane < nr) cl.map_shared_rank(sm.xw, q)[r0 + lane] = w;
                if (lane == 0) cl.map_shared_rank(sm.xn, q)[rank] = n2;
            }
        }
        cl.sync();
        double b2 = 0.0;
        for (int q = 0; q < SK_CL; ++q) b2 += sm.xn[q];
        const double bj = sqrt(b2);
        if (warp == 0) {
            const double al = sm.h1[j].x + sm.h2[j].x;
            if (lane == 0) {
                sm.beta[j] = bj;
                sm.alpha[j] = al;
            }
            if (arnoldi)   // the whole column j: projections, beta_j, zeros below
                sm.hess[32 * j + lane] = lane <= j ? cadd(sm.h1[lane], sm.h2[lane])
                                                   : make_double2(lane == j + 1 ? bj : 0.0, 0.0);
            __syncwarp();
            if (arnoldi) hess_expm_warp(sm.hess, sm.hvec, j + 1, zr, zi, sm.c);
            else tridiag_expm_warp(sm.alpha, sm.beta, j + 1, zr, zi, sm.c);
            __syncwarp();
            if (lane == 0) {
                const cplx cj = sm.c[j];
                const double err = bj * sqrt(cj.x * cj.x + cj.y * cj.y);
                sm.conv = err <= tol;
                if (!isfinite(err) || !isfinite(al)) sm.nonfin = 1;
                sm.done = sm.conv || sm.nonfin || j == mmax - 1;
                sm.err = err;
            }
        } else {
            // meanwhile: v_{j+1} and its product (not used when this step was the last)
            const double inv = bj > 0.0 ? 1.0 / bj : 0.0;
            cplx* vn = V + (j + 1) * s;
            for (int e = tid - 32; e < s; e += SK_THREADS - 32) vn[e] = make_double2(sm.xw[e].x * inv, sm.xw[e].y * inv);
            asm volatile("bar.sync 1, %0;" ::"n"(SK_THREADS - 32) : "memory");
            matvec(vn, tid - 32, SK_THREADS - 32);
        }
        __syncthreads();
        if (sm.done) break;
    }
    // x = |x0| sum_i c_i v_i, own rows
    if (tid < nr) {
        cplx acc = make_double2(0.0, 0.0);
        for (int i = 0; i <= j; ++i) acc_cmul(acc, V[i * s + r0 + tid], sm.c[i]);
        x[r0 + tid] = make_double2(acc.x * nrm0, acc.y * nrm0);
    }
    if (rank == 0 && tid == 0) {
        KrylovStatus& st = pub.hs->krylov[0];
        st.err = sm.err;
        st.converged = sm.conv;
        st.nonfinite = sm.nonfin;
        st.iters = j + 1;
        publish(pub);
    }
}

__global__ void permute3_kernel(const cplx* x, cplx* y, int d0, int d1, int d2, int p0, int p1, int p2,
                                int inverse) {
    pdl_begin();
    // y has axes (x-axis p0, x-axis p1, x-axis p2), first fastest
    long long n = (long long)d0 * d1 * d2;
    int dims[3] = {d0, d1, d2};
    int q[3] = {p0, p1, p2};
    int e0 = dims[q[0]], e1 = dims[q[1]];
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        long long i0 = e % e0, r = e / e0;
        long long i1 = r % e1, i2 = r / e1;
        long long idx[3];
        idx[q[0]] = i0;
        idx[q[1]] = i1;
        idx[q[2]] = i2;
        long long src = idx[0] + (long long)d0 * (idx[1] + (long long)d1 * idx[2]);
        if (!inverse) y[e] = x[src];
        else y[src] = x[e];
    }
}

__global__ void fill_kernel(cplx* x, long long n, cplx v) {
    pdl_begin();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        x[e] = v;
}

// H = Hs + sum over sites and driven atoms, coef: 5 doubles per atom
// (omega_x, omega_z, Re W, Im W, delta).  Most coefficients of a pulse layer are
// zero at a given time, and one thread per entry walking all atoms was a serial
// chain of loads (16 us for a 12 x 12 block of 62 atoms): the block first
// lists the terms whose coefficients are not all zero and reads only their
// operators, several in flight.  Terms are added one by one in atom order.
// Measured, us per block (8x8 lattice, chi = 12): 15.8 -> 8.0.
constexpr int AB_THREADS = 128;
__global__ void __launch_bounds__(AB_THREADS)
    assemble_block_kernel(cplx* H, const cplx* Hs, int D, const cplx* nops, int nsites, const int* site_ids,
                          const cplx* dops, int ndriven, const int* driven_ids, const double* coef, double gamma) {
    pdl_begin();
    extern __shared__ short terms[];       // < nsites: site term, else driven atom (index - nsites)
    __shared__ int s_count;
    if (threadIdx.x < 32) {                // in order, by one warp
        int count = 0;
        const int n = nsites + ndriven;
        for (int b = 0; b < n; b += 32) {
            const int i = b + threadIdx.x;
            bool on = false;
            if (i < nsites) {
                on = gamma != 0.0 || coef[5 * site_ids[i] + 4] != 0.0;
            } else if (i < n) {
                const double* c = coef + 5 * driven_ids[i - nsites];
                on = c[0] != 0.0 || c[1] != 0.0 || c[2] != 0.0 || c[3] != 0.0;
            }
            const unsigned m = __ballot_sync(0xffffffffu, on);
            if (on) terms[count + __popc(m & ((1u << threadIdx.x) - 1u))] = (short)i;
            count += __popc(m);
        }
        if (threadIdx.x == 0) s_count = count;
    }
    __syncthreads();
    const int count = s_count;
    const long long DD = (long long)D * D;
    for (long long e = blockIdx.x * (long long)AB_THREADS + threadIdx.x; e < DD; e += (long long)gridDim.x * AB_THREADS) {
        const int a = (int)(e % D), b = (int)(e / D);
        const long long et = b + (long long)D * a;           // transposed position
        cplx h = Hs ? Hs[e] : make_double2(0.0, 0.0);
        int i = 0;
#pragma unroll 4
        for (; i < count && terms[i] < nsites; ++i) {
            // -(Delta_i + i gamma) n_i: detuning, and the decay of Eq. 3
            const int q = terms[i];
            const double de = coef[5 * site_ids[q] + 4];
            const cplx v = nops[q * DD + e];
            h.x -= de * v.x - gamma * v.y;
            h.y -= de * v.y + gamma * v.x;
        }
#pragma unroll 2
        for (; i < count; ++i) {
            const int q = terms[i] - nsites;
            const double* c = coef + 5 * driven_ids[q];
            const cplx* sx = dops + (3LL * q) * DD;
            cplx t = make_double2(0.0, 0.0);
            if (c[0] != 0.0) {
                const cplx v = sx[e];
                t.x = c[0] * v.x;
                t.y = c[0] * v.y;
            }
            if (c[1] != 0.0) {
                const cplx v = sx[DD + e];
                t.x = fma(c[1], v.x, t.x);
                t.y = fma(c[1], v.y, t.y);
            }
            if (c[2] != 0.0 || c[3] != 0.0) {
                // W rp + conj(W) rp^H ; rp^H(a, b) = conj(rp(b, a))
                const cplx vr = sx[2 * DD + e], vt = sx[2 * DD + et];
                t.x = t.x + (c[2] * vr.x - c[3] * vr.y) + (c[2] * vt.x - c[3] * vt.y);
                t.y = t.y + (c[2] * vr.y + c[3] * vr.x) + (-c[2] * vt.y - c[3] * vt.x);
            }
            h.x += t.x;
            h.y += t.y;
        }
        H[e] = h;
    }
}

__global__ void check_finite_kernel(const cplx* x, long long n, int* flag) {
    pdl_begin();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        cplx v = x[e];
        if (!isfinite(v.x) || !isfinite(v.y)) flag[0] = 1;
    }
}

// G_i = sum_j W[j + nb*i] N_j for i < r (real weights, complex matrices of n
// entries each, stacked contiguously): the channel operators
// G_i = sum_j V_ij n_j of an effective Hamiltonian.  One thread per matrix
// entry keeps up to 16 outputs in registers and reads each N_j entry once per
// group of 16 outputs (memory bound for the few outputs of a group).
template <int WSUM_GROUP>
__global__ void weighted_sum_kernel(const cplx* __restrict__ N, int nb, long long n, const double* __restrict__ W,
                                    int r, cplx* __restrict__ G, int staged) {
    pdl_begin();
    extern __shared__ double sw_smem[];
    const double* sw = W;   // weights from global memory unless they fit in shared memory
    if (staged) {
        for (int i = threadIdx.x; i < nb * r; i += blockDim.x) sw_smem[i] = W[i];
        __syncthreads();
        sw = sw_smem;
    }
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        for (int i0 = 0; i0 < r; i0 += WSUM_GROUP) {
            cplx acc[WSUM_GROUP];
#pragma unroll
            for (int t = 0; t < WSUM_GROUP; ++t) acc[t] = make_double2(0.0, 0.0);
#pragma unroll 4
            for (int j = 0; j < nb; ++j) {   // unrolled: several loads in flight per thread
                const cplx v = N[(long long)j * n + e];
#pragma unroll
                for (int t = 0; t < WSUM_GROUP; ++t) {
                    if (i0 + t < r) {
                        const double w = sw[j + nb * (i0 + t)];
                        acc[t].x = fma(w, v.x, acc[t].x);
                        acc[t].y = fma(w, v.y, acc[t].y);
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < WSUM_GROUP; ++t)
                if (i0 + t < r) G[(long long)(i0 + t) * n + e] = acc[t];
        }
    }
}

// The same for few outputs (entries times r): S threads per output share the
// sum over j (62 loads in a row took 30 us for a 9 x 9 stack, 7 now).
template <int S>
__global__ void __launch_bounds__(128) weighted_sum_small_kernel(const cplx* __restrict__ N, int nb, int n,
                                                                 const double* __restrict__ W, int r,
                                                                 cplx* __restrict__ G) {
    pdl_begin();
    constexpr int OB = 128 / S;
    __shared__ cplx part[128];
    const int o = threadIdx.x % OB, ks = threadIdx.x / OB;
    const int out = blockIdx.x * OB + o, e = out % n, i = out / n;
    cplx acc = make_double2(0.0, 0.0);
    if (i < r) {
#pragma unroll 4
        for (int j = ks; j < nb; j += S) {
            const cplx v = N[(long long)j * n + e];
            const double w = W[j + nb * i];
            acc.x = fma(w, v.x, acc.x);
            acc.y = fma(w, v.y, acc.y);
        }
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    if (ks != 0 || i >= r) return;
#pragma unroll
    for (int q = 1; q < S; ++q) acc = cadd(acc, part[q * OB + o]);
    G[(long long)i * n + e] = acc;
}

// FP64 throughput probes: many independent FMA chains per thread (the FP64
// ALU, DFMA), or chains of FP64 tensor-core instructions (DMMA,
// mma.sync m8n8k4 f64; four independent accumulators per warp).  The result
// is stored only under a condition that never holds, which keeps the
// compiler from removing the chains.
constexpr int PROBE_CHAINS = 8;
__global__ void fp64_fma_probe_kernel(double* out, int iters) {
    double a[PROBE_CHAINS];
#pragma unroll
    for (int k = 0; k < PROBE_CHAINS; ++k) a[k] = 1e-9 * (threadIdx.x + k);
    const double b = 0.999999999, c = 1e-12;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < PROBE_CHAINS; ++k) a[k] = fma(a[k], b, c);
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < PROBE_CHAINS; ++k) s += a[k];
    if (s == 12345.678) out[0] = s;
}

__global__ void dmma_probe_kernel(double* out, int iters) {
    const double a = 1e-9 * (threadIdx.x & 31), b = 0.5;
    double d[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k][0] = d[k][1] = 0.0;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                         : "+d"(d[k][0]), "+d"(d[k][1])
                         : "d"(a), "d"(b));
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) s += d[k][0] + d[k][1];
    if (s == 12345.678) out[0] = s;
}

inline int grid_for(long long n) {
    long long g = (n + 255) / 256;
    if (g > 4 * 152) g = 4 * 152;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

// ------------------------------------------------------------------ launchers
int red_blocks_for(long long n) {
    // 64 elements per block while blocks are free: a 6561-entry node on four
    // blocks of 2048 left 148 SMs idle on FP64-bound sums
    long long g = (n + 63) / 64;
    if (g > RED_BLOCKS) g = RED_BLOCKS;
    if (g < 1) g = 1;
    return (int)g;
}

int k_norm2_partial(const cplx* x, long long n, double* partial, cudaStream_t s) {
    int G = red_blocks_for(n);
    launch(norm2_partial_kernel, G, T, 0, s, x, n, G, partial);
    return 1;
}

int k_dots(const cplx* V, long long ld, int nv, const cplx* w, long long n, cplx* partial, cudaStream_t s) {
    const int G = red_blocks_for(n);
    launch(dots_kernel, G, T, 0, s, V, ld, nv, w, n, G, partial);
    return 1;
}

int k_orth_first(const cplx* V, long long ld, int nv, const cplx* partial_in, cplx* w, long long n, cplx* partial_dots,
                 cplx* h_out, cudaStream_t s) {
    const int G = red_blocks_for(n);
    launch(orth_first_kernel, G, T, 0, s, V, ld, nv, partial_in, w, n, G, partial_dots, h_out);
    return 1;
}

int k_lanczos_first(const cplx* V, long long ld, int j, const cplx* partial_in, const KrylovScalars* ks, cplx* w,
                    long long n, cplx* partial_dots, cplx* h_out, cudaStream_t s) {
    const int G = red_blocks_for(n);
    launch(lanczos_first_kernel, G, T, 0, s, V, ld, j, partial_in, ks, w, n, G, partial_dots, h_out);
    return 1;
}

int k_orth_second(const cplx* V, long long ld, int nv, const cplx* partial_in, cplx* w, long long n,
                  double* partial_norm, KrylovScalars* ks, const cplx* h1, double zr, double zi, double tol,
                  int arnoldi, const Publish& pub, cudaStream_t s) {
    const int G = red_blocks_for(n);
    launch(orth_second_kernel, G, T, 0, s, V, ld, nv, partial_in, w, n, G, partial_norm, ks, h1, zr, zi, tol, arnoldi,
           pub);
    return 1;
}

int k_scale_copy_dev(const cplx* x, long long n, const double* scale, cplx* y, cudaStream_t s) {
    launch(scale_copy_kernel, grid_for(n), 256, 0, s, x, n, scale, y);
    return 1;
}

int k_rescale_to_norm(cplx* x, long long n, const double* px, int Gx, const double* pr, int Gr, cudaStream_t s) {
    launch(rescale_to_norm_kernel, grid_for(n), 256, 0, s, x, n, px, Gx, pr, Gr);
    return 1;
}

int k_combine(const cplx* V, long long ld, int nv, const KrylovScalars* ks, cplx* y, long long n,
              cudaStream_t s) {
    launch(combine_kernel, grid_for(n), 256, 0, s, V, ld, nv, ks, y, n);
    return 1;
}

int k_krylov_start(KrylovScalars* ks, const cplx* x, long long n, double* partial, cudaStream_t s) {
    const int G = red_blocks_for(n);
    launch(krylov_start_kernel, G, T, 0, s, ks, x, n, G, partial, &ks->arrived);
    return 1;
}

bool wait_status(const HostStatus* hs, unsigned seq, cudaStream_t s) {
    const volatile unsigned* p = &hs->seq;
    auto there = [&] { return (int)(*p - seq) >= 0; };
    unsigned schedule = cudaDeviceScheduleAuto;
    for (unsigned i = 1;; ++i) {
        if (there()) break;
        if ((i & 0xFFF) != 0) continue;
        // a long wait (some 10 us): as the device's scheduling flag has it, and
        // look whether the stream is done or has failed
        if (i == 0x1000) {
            if (cudaGetDeviceFlags(&schedule) != cudaSuccess) cudaGetLastError();
            schedule &= cudaDeviceScheduleMask;
        }
        if (schedule == cudaDeviceScheduleYield) sched_yield();
        if (schedule == cudaDeviceScheduleBlockingSync ? cudaStreamSynchronize(s) != cudaErrorNotReady
                                                       : cudaStreamQuery(s) != cudaErrorNotReady) {
            if (there()) break;
            return false;
        }
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    return true;
}

int k_permute3(const cplx* x, cplx* y, int d0, int d1, int d2, int p0, int p1, int p2, int inverse,
               cudaStream_t s) {
    long long n = (long long)d0 * d1 * d2;
    launch(permute3_kernel, grid_for(n), 256, 0, s, x, y, d0, d1, d2, p0, p1, p2, inverse);
    return 1;
}

int k_fill(cplx* x, long long n, cplx v, cudaStream_t s) {
    if (n <= 0) return 0;
    launch(fill_kernel, grid_for(n), 256, 0, s, x, n, v);
    return 1;
}

int k_assemble_block(cplx* H, const cplx* Hs, int D, const cplx* nops, int nsites, const int* site_ids,
                     const cplx* dops, int ndriven, const int* driven_ids, const double* coef, double gamma,
                     cudaStream_t s) {
    long long DD = (long long)D * D;
    const size_t smem = sizeof(short) * (size_t)std::max(1, nsites + ndriven);
    launch(assemble_block_kernel, (unsigned)std::min<long long>((DD + AB_THREADS - 1) / AB_THREADS, 8 * 152),
           AB_THREADS, smem, s, H, Hs, D, nops, nsites, site_ids, dops, ndriven, driven_ids, coef, gamma);
    return 1;
}

int k_check_finite(const cplx* x, long long n, int* flag, cudaStream_t s) {
    if (n <= 0) return 0;
    launch(check_finite_kernel, grid_for(n), 256, 0, s, x, n, flag);
    return 1;
}

// FP64 peak probe (method 0: DFMA chains, 1: DMMA m8n8k4): launches one probe
// over `blocks` blocks of 256 threads and returns its flop count; the caller
// times it.  2 flops per FMA; 2 * 8 * 8 * 4 flops per warp-wide DMMA.
double k_fp64_probe(int method, int blocks, int iters, double* out, cudaStream_t s) {
    if (method == 0) {
        fp64_fma_probe_kernel<<<blocks, 256, 0, s>>>(out, iters);
        return 2.0 * PROBE_CHAINS * (double)iters * 256.0 * blocks;
    }
    dmma_probe_kernel<<<blocks, 256, 0, s>>>(out, iters);
    return 512.0 * 4.0 * (double)iters * (256.0 / 32.0) * blocks;
}

int k_weighted_sum(const cplx* N, int nb, long long n, const double* W, int r, cplx* G, cudaStream_t s) {
    if (n <= 0 || r <= 0) return 0;
    if (n * r <= 64 * 1024) {   // below that the chip is not full with one thread per entry
        const int outs = (int)(n * r);
        if (nb >= 32 && outs <= 16 * 1024) launch(weighted_sum_small_kernel<16>, (outs + 7) / 8, 128, 0, s, N, nb,
                                                  (int)n, W, r, G);
        else if (nb >= 4) launch(weighted_sum_small_kernel<4>, (outs + 31) / 32, 128, 0, s, N, nb, (int)n, W, r, G);
        else launch(weighted_sum_small_kernel<1>, (outs + 127) / 128, 128, 0, s, N, nb, (int)n, W, r, G);
        return 1;
    }
    const size_t need = sizeof(double) * (size_t)nb * r;
    const int staged = need <= 48 * 1024;
    // small blocks: the work per entry is nb * r FP64 FMAs, so spread the
    // entries over every SM
    const long long blocks = std::min<long long>((n + 63) / 64, 16 * 152);
    if (r <= 4)   // few outputs: small register groups, more loads in flight
        launch(weighted_sum_kernel<4>, (unsigned)blocks, 64, staged ? need : 0, s, N, nb, n, W, r, G, staged);
    else
        launch(weighted_sum_kernel<16>, (unsigned)blocks, 64, staged ? need : 0, s, N, nb, n, W, r, G, staged);
    return 1;
}

int k_small_krylov(const int* d, const cplx* hb0, const cplx* hb1, const cplx* hb2, const SmallPairs& pp, cplx* x,
                   double zr, double zi, double tol, int mmax, int arnoldi, const Publish& pub, cudaStream_t s) {
    const int n = d[0] * d[1] * d[2], R = (n + SK_CL - 1) / SK_CL;
    const size_t smem = sizeof(cplx) * ((size_t)R * n + (size_t)(mmax + 1) * n);
    // the shared-memory limit is a per-device attribute of the kernel: set it
    // once on every device the process uses
    static std::mutex mu;
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!attr[dev]) {
            cudaFuncSetAttribute(small_krylov_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(cplx) *
                                       ((size_t)SK_ROWS * SMALL_S + (size_t)(KRYLOV_MMAX + 1) * SMALL_S)));
            attr[dev] = true;
        }
    }
    launch(small_krylov_kernel, SK_CL, SK_THREADS, smem, s, d[0], d[1], d[2], hb0, hb1, hb2, pp, x, zr, zi, tol, mmax,
           arnoldi, pub);
    return 1;
}
