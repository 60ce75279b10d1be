// QR of a tall, well-conditioned node matricisation by panels of 32 columns:
// block Gram-Schmidt with Cholesky factors of Gram matrices, every pass over
// the rows a contraction on the tensor cores (gemm_digits.cu).
// First every column is scaled by a power of two to a norm in [1, 2)
// (exactly), then per panel W (Q: the columns before it, final), twice:
//   S = [Q W]^H W,   G = S_w - S_q^H S_q = L L^H   (Gram of W without its part along Q),
//   W <- (W - Q S_q) L^-H = [Q W] [-S_q L^-H ; L^-H].
// The second time W is orthonormal up to the square of the first pass's
// condition number times 2^-53, and the repetition brings it to rounding
// (Carson, Lund, Rozloznik, Thomas, "Block Gram-Schmidt algorithms and their
// stability properties", Linear Algebra Appl. 638, 2022: BCGS-PIP+).  At the end
// R = Q^H A with the unscaled A.
//
// Accuracy.  A digit contraction holds a row of its operand on one grid, 2^-55 of
// the row's largest entry, so the rows of [Q W] are only held well if Q and W
// are of one size: unscaled, W lost 1e-15 / |A| of itself (1e-9 of a matrix of
// norm 1e-6).  Scaled, |Q R - A| is below 1e-15 of every column on its own scale
// (the column loop: 2e-16).  R multiplied up from the passes' factors instead of
// Q^H A lost up to the panel's condition number times 2^-55 (1e-13 of a column
// 2e-4 away from the span of the others); the product costs 0.16 ms of 16384 x 128
// (1.86 -> 2.02).
//
// The column-by-column rule (qr.cu) decides which columns are dependent; this
// path is for matrices without any: it gives up (the flag) as soon as a
// column's part outside the earlier ones is below 1e-4 of the column or 1e-8
// of |A|_F, far above the rule's 1e-10, and when |A| lies outside 2^+-480, and the
// caller runs the column loop on the original matrix; what has been launched
// beyond that point does nothing.  Q and R are then the same as the column loop's up to rounding (R has
// a positive real diagonal, which makes them unique).
//
// Why: 16 M D^2 flops of the column loop take 4.1 ms on the FP64 pipe for a
// 16384 x 128 matrix, and its 128 columns as many grid synchronisations
// (8.5 ms measured); here the rows are read by ~10 launches per panel and
// pass.  Measured, ms per call, column loop (with its rows spread over all SMs)
// and panels: 16384 x 128 7.5 and 2.0, 10368 x 81 2.9 and 1.17, 6561 x 128 4.2
// and 1.48, 4096 x 64 1.25 and 0.67, 81 x 81 1.1 and 0.79.
#include "common.cuh"

#include <algorithm>
#include <cstring>

namespace {

constexpr int PB = QR_PANEL;       // panel width
constexpr int CT = 512;            // threads of the Cholesky kernel
constexpr double MIN_COL2 = 1e-8;  // residual^2 / |column|^2
constexpr double MIN_FRO2 = 1e-16; // residual^2 / |A|_F^2
constexpr double DEP_COL2 = 1e-14; // below: as good as a dependent column (flag 2)
constexpr int MAX_EXP = 480;       // |A| = 2^+-480 and beyond: squares leave the FP64 range
constexpr int ST = 512;            // threads of the scaling kernel
constexpr int FT = 1024;           // threads of the finishing kernel

// Column b of A to W as x 2^-e with a norm in [1, 2): cexp[b] = e, norm2[b] the
// squared norm of the scaled column.  Zero columns and columns with an infinity
// or a NaN are copied as they are.  One block per column; the column is read
// three times (largest exponent, norm, copy), the second and third time from
// L2: 9 us for 16384 x 128, as a plain copy and the norm of A took before.
__global__ void __launch_bounds__(ST) panel_scale_kernel(const cplx* A, int M, cplx* W, double* norm2, int* cexp) {
    pdl_begin();
    const cplx* a = A + (long long)blockIdx.x * M;
    cplx* w = W + (long long)blockIdx.x * M;
    __shared__ int s_max;
    __shared__ double part[ST / 32];
    const int t = threadIdx.x;
    if (t == 0) s_max = 0;
    __syncthreads();
    int m = 0;
#pragma unroll 4
    for (int i = t; i < M; i += ST) {
        const cplx x = a[i];
        const unsigned hx = (unsigned)__double2hiint(x.x) & 0x7FFFFFFFu, hy = (unsigned)__double2hiint(x.y) & 0x7FFFFFFFu;
        m = max(m, (int)(max(hx, hy) >> 20));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((t & 31) == 0) atomicMax(&s_max, m);
    __syncthreads();
    const int e0 = s_max == 0 || s_max == 0x7FF ? 0 : s_max - 1022;   // entries below 2^e0
    const double f0 = scalbn(1.0, -e0);
    double s = 0.0;
#pragma unroll 4
    for (int i = t; i < M; i += ST) {
        const cplx x = a[i];
        s = fma(x.x * f0, x.x * f0, fma(x.y * f0, x.y * f0, s));
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((t & 31) == 0) part[t >> 5] = s;
    __syncthreads();
    s = 0.0;
    for (int q = 0; q < ST / 32; ++q) s += part[q];
    int e1 = 0;
    if (s > 0.0 && isfinite(s)) e1 = (ilogb(s) + 2048) / 2 - 1024;   // floor(log2(norm))
    const double f = scalbn(1.0, -(e0 + e1));
#pragma unroll 4
    for (int i = t; i < M; i += ST) {
        const cplx x = a[i];
        w[i] = make_double2(x.x * f, x.y * f);
    }
    if (t == 0) {
        norm2[blockIdx.x] = scalbn(s, -2 * e1);
        cexp[blockIdx.x] = e0 + e1;
    }
}

// G = Sw + Gq (bp x bp, Hermitian; Sw with leading dimension ld, Gq with PB,
// nullptr: none) = L L^H; T = L^-H into rows [n, n + bp) of C (leading
// dimension ld).  One block: right-looking Cholesky, the same eliminations
// applied to the identity give L^-1.  pass 2 expects a matrix near the
// identity.  Sets *flag when a pivot is too small (2: down to rounding): cn2, cexp are the squared
// norms and exponents of all D scaled columns, the panel's first is column n.
__global__ void __launch_bounds__(CT) panel_chol_kernel(const cplx* Sw, long long ld, const cplx* Gq, int bp, cplx* C,
                                                        const double* cn2, const int* cexp, int D, int n, int pass,
                                                        int* flag) {
    pdl_begin();
    __shared__ cplx G[PB][PB + 1], X[PB][PB + 1];
    __shared__ double norm2[PB], floor2[PB], s_inv;
    __shared__ int bad;
    const int t = threadIdx.x;
    if (*(volatile int*)flag) return;   // an earlier panel gave up
    if (t == 0) bad = 0;
    if (pass == 1 && t < 32) {   // |A|_F^2 in units of 4^top, then the least residual^2 of each scaled column
        int top = -(1 << 20);
        for (int k = t; k < D; k += 32) top = max(top, cexp[k]);
        top = __reduce_max_sync(0xffffffffu, top);
        double f = 0.0;
        for (int k = t; k < D; k += 32) f += scalbn(cn2[k], 2 * (cexp[k] - top));
        for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
        if (t < bp) floor2[t] = scalbn(MIN_FRO2 * f, 2 * (top - cexp[n + t]));
        if (t == 0 && (top > MAX_EXP || top < -MAX_EXP)) bad = 1;
    }
    for (int e = t; e < PB * PB; e += CT) {
        const int i = e % PB, j = e / PB;
        cplx g = make_double2(i == j ? 1.0 : 0.0, 0.0);
        if (i < bp && j < bp) {
            g = Sw[i + j * ld];
            if (i == j) norm2[i] = g.x;
            if (Gq) {
                const cplx q = Gq[i + j * PB];
                g.x += q.x;
                g.y += q.y;
            }
            if (i == j) g.y = 0.0;
        }
        G[i][j] = g;
        X[i][j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    for (int k = 0; k < bp; ++k) {
        if (t == 0) {
            const double d = G[k][k].x;
            const bool ok = pass == 1 ? (d >= MIN_COL2 * norm2[k] && d > floor2[k]) : d >= 0.25;
            if (!ok || !isfinite(d)) bad = pass == 1 && d <= DEP_COL2 * norm2[k] ? 2 : 1;
            s_inv = rsqrt(d);
        }
        __syncthreads();
        if (bad) {
            if (t == 0) *flag = bad;
            return;
        }
        const double inv = s_inv;
        if (t < PB) {
            if (t > k) {
                G[t][k].x *= inv;
                G[t][k].y *= inv;
            } else {
                X[k][t].x *= inv;
                X[k][t].y *= inv;
            }
        }
        __syncthreads();
        for (int e = t; e < (PB - 1 - k) * PB; e += CT) {
            // G_ij -= l_ik conj(l_jk) (j > k), X_ij -= l_ik x_kj (j <= k): one
            // instruction stream for both
            const int i = k + 1 + e / PB, j = e % PB;
            if (j > i) continue;
            const cplx l = G[i][k];
            cplx m = j > k ? G[j][k] : X[k][j];
            if (j > k) m.y = -m.y;
            cplx* z = j > k ? &G[i][j] : &X[i][j];
            cplx g = *z;
            g.x = fma(-l.x, m.x, fma(l.y, m.y, g.x));
            g.y = fma(-l.x, m.y, fma(-l.y, m.x, g.y));
            *z = g;
        }
        __syncthreads();
    }
    for (int e = t; e < bp * bp; e += CT) {
        const int i = e % bp, j = e / bp;   // upper triangular: T = X^H
        C[i + j * ld] = i <= j ? make_double2(X[j][i].x, -X[j][i].y) : make_double2(0.0, 0.0);
    }
}

__device__ __forceinline__ void panel_publish(const Publish& pub, int flag) {
    if (!pub.hs) return;
    pub.hs->qr_flag = flag;
    if (pub.tc_flag && *(volatile const int*)pub.tc_flag) pub.hs->tc_flag = 1;
    __threadfence_system();
    *(volatile unsigned*)&pub.hs->seq = pub.seq;
}

__global__ void panel_report_kernel(const int* flag, Publish pub) {
    pdl_begin();
    panel_publish(pub, *flag);
}

// By a whole block, col2 and diag (of D) in shared memory: squared column
// norms and the diagonal of the upper triangular R.  A warp per column; tidy:
// clear what is below the diagonal and the diagonal's imaginary part first.
__device__ void r_columns(cplx* R, int D, bool tidy, double* col2, double* diag) {
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < D; k += FT / 32) {
        cplx* r = R + (long long)k * D;
        double s = 0.0;
        for (int i = lane; i < (tidy ? D : k + 1); i += 32) {
            cplx x = r[i];
            if (i > k) x = make_double2(0.0, 0.0);
            if (i == k) {
                x.y = 0.0;
                diag[k] = x.x;
            }
            if (tidy && i >= k) r[i] = x;
            s = fma(x.x, x.x, fma(x.y, x.y, s));
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) col2[k] = s;
    }
    __syncthreads();
}

// By one warp: does a diagonal entry lie below `margin` times the limits?
__device__ bool r_refused(const double* col2, const double* diag, int D, double margin) {
    const int lane = threadIdx.x & 31;
    double f = 0.0;
    for (int k = lane; k < D; k += 32) f += col2[k];
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    bool bad = false;
    for (int k = lane; k < D; k += 32) {
        const double d = diag[k], d2 = d * d;
        if (!(d > 0.0 && d2 >= margin * MIN_COL2 * col2[k] && d2 > margin * MIN_FRO2 * f)) bad = true;
    }
    return __any_sync(0xffffffffu, bad);
}

// R = Q^H A made upper triangular with a real diagonal, and the residuals
// checked once more on the final R (the Gram matrices know them less well).
// One block.
__global__ void __launch_bounds__(FT) panel_finish_kernel(cplx* R, int D, int* flag, Publish pub) {
    pdl_begin();
    __shared__ double col2[256], diag[256];
    const int gave_up = *(volatile int*)flag;   // R has not been written
    __syncthreads();
    if (!gave_up) r_columns(R, D, true, col2, diag);
    if (threadIdx.x >= 32) return;
    const int bad = gave_up ? gave_up : (int)r_refused(col2, diag, D, 1.0);
    if (threadIdx.x == 0) panel_publish(pub, bad);
}

// The final check on another QR's R: its diagonal agrees with the panels' to
// 1e-11 at the limits (2^-53 |a| against 1e-4 |a|), so what is below 0.9 of them is
// refused for certain.  One block.
__global__ void __launch_bounds__(FT) panel_verdict_kernel(cplx* R, int D, Publish pub) {
    pdl_begin();
    __shared__ double col2[256], diag[256];
    r_columns(R, D, false, col2, diag);
    if (threadIdx.x >= 32) return;
    const bool bad = r_refused(col2, diag, D, 0.9);
    if (threadIdx.x == 0) panel_publish(pub, bad);
}

GemmArgs args(int M, int N, int K) {
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = M;
    g.N = N;
    g.Ki = K;
    g.Ko = g.Bi = g.Bo = 1;
    g.alpha = make_double2(1.0, 0.0);
    return g;
}

GemmArgs gram_args(const cplx* A, int M, int n, int bp, cplx* S) {   // S = [Q W]^H W
    GemmArgs g = args(n + bp, bp, M);
    g.A = A; g.a_m = M; g.a_ki = 1; g.conjA = 1;
    g.B = A + (long long)n * M; g.b_ki = 1; g.b_n = M;
    g.C = S; g.c_m = 1; g.c_n = n + bp;
    return g;
}

GemmArgs r_args(const cplx* Q, const cplx* A, int M, int D, cplx* R) {   // R = Q^H A
    GemmArgs g = args(D, D, M);
    g.A = Q; g.a_m = M; g.a_ki = 1; g.conjA = 1;
    g.B = A; g.b_ki = 1; g.b_n = M;
    g.C = R; g.c_m = 1; g.c_n = D;
    return g;
}

GemmArgs update_args(cplx* A, int M, int n, int bp, const cplx* C) {   // W = [Q W] C, in place
    GemmArgs g = args(M, bp, n + bp);
    g.A = A; g.a_m = 1; g.a_ki = M;
    g.B = C; g.b_ki = 1; g.b_n = n + bp;
    g.C = A + (long long)n * M; g.c_m = 1; g.c_n = M;
    return g;
}

}  // namespace

size_t qr_panel_scratch(int D) {   // complex: S and C, Gq, column norms and exponents
    return 2 * (size_t)(D + PB) * PB + PB * PB + D;
}

size_t qr_panel_workspace(int M, int D) {
    size_t need = digits_workspace_bytes(r_args(nullptr, nullptr, M, D, nullptr), false);
    for (int n = 0; n < D; n += PB) {
        const int bp = std::min(PB, D - n);
        need = std::max(need, std::max(digits_workspace_bytes(gram_args(nullptr, M, n, bp, nullptr), false),
                                       digits_workspace_bytes(update_args(nullptr, M, n, bp, nullptr), false)));
    }
    return need;
}

int qr_panel(const cplx* A, cplx* Q, int M, int D, cplx* R, QrScratch& ws, cudaStream_t s, void* workspace,
             size_t workspace_bytes, int first, int last, const Publish& pub) {
    cplx* S = ws.panel;
    cplx* C = S + (long long)(D + PB) * PB;
    cplx* Gq = C + (long long)(D + PB) * PB;
    double* cn2 = reinterpret_cast<double*>(Gq + PB * PB);
    int* cexp = reinterpret_cast<int*>(cn2 + D);
    int* flag = ws.err + 1;
    int launches = 0;
    if (first == 0) {
        if (cudaMemsetAsync(flag, 0, sizeof(int), s) != cudaSuccess) return -1;
        launch(panel_scale_kernel, D, ST, 0, s, A, M, Q, cn2, cexp);
        ++launches;
    }
    last = std::min(D, last);
    for (int n = first; n < last; n += PB) {
        const int bp = std::min(PB, D - n), ld = n + bp;
        for (int pass = 1; pass <= 2; ++pass) {
            int l = launch_zgemm_digits(gram_args(Q, M, n, bp, S), false, s, workspace, workspace_bytes, flag);
            if (l < 0) return -1;
            launches += l;
            if (n > 0) {   // -S_q^H S_q
                GemmArgs g = args(bp, bp, n);
                g.A = S; g.a_m = ld; g.a_ki = 1; g.conjA = 1;
                g.B = S; g.b_ki = 1; g.b_n = ld;
                g.C = Gq; g.c_m = 1; g.c_n = PB;
                g.alpha = make_double2(-1.0, 0.0);
                launches += launch_zgemm_f64(g, s);
            }
            launch(panel_chol_kernel, 1, CT, 0, s, S + n, ld, n > 0 ? Gq : nullptr, bp, C + n, cn2, cexp, D, n, pass,
                   flag);
            ++launches;
            if (n > 0) {   // -S_q T
                GemmArgs g = args(n, bp, bp);
                g.A = S; g.a_m = 1; g.a_ki = ld;
                g.B = C + n; g.b_ki = 1; g.b_n = ld;
                g.C = C; g.c_m = 1; g.c_n = ld;
                g.alpha = make_double2(-1.0, 0.0);
                launches += launch_zgemm_f64(g, s);
            }
            // in place: the operands are packed before the first output is written
            l = launch_zgemm_digits(update_args(Q, M, n, bp, C), false, s, workspace, workspace_bytes, flag);
            if (l < 0) return -1;
            launches += l;
        }
    }
    if (last < D) {
        launch(panel_report_kernel, 1, 1, 0, s, flag, pub);
        return launches + 1;
    }
    const int l = launch_zgemm_digits(r_args(Q, A, M, D, R), false, s, workspace, workspace_bytes, flag);
    if (l < 0) return -1;
    launch(panel_finish_kernel, 1, FT, 0, s, R, D, flag, pub);
    return launches + l + 1;
}

int qr_panel_verdict(const cplx* R, int D, cudaStream_t s, const Publish& pub) {
    launch(panel_verdict_kernel, 1, FT, 0, s, const_cast<cplx*>(R), D, pub);
    return 1;
}
