// QR of a tall, well-conditioned node matricisation by panels of 32 columns:
// block Gram-Schmidt with Cholesky factors of Gram matrices, every pass over
// the rows a contraction on the tensor cores (gemm_digits.cu, FP64 results).
// Per panel W (Q: the columns before it, final), twice:
//   S = [Q W]^H W,   G = S_w - S_q^H S_q = L L^H   (Gram of W without its part along Q),
//   W <- (W - Q S_q) L^-H = [Q W] [-S_q L^-H ; L^-H].
// The second time W is orthonormal up to the square of the first pass's
// condition number times 2^-53, and the repetition brings it to rounding
// (Carson, Lund, Rozloznik, Thomas, "Block Gram-Schmidt algorithms and their
// stability properties", Linear Algebra Appl. 638, 2022: BCGS-PIP+).  R's
// panel is S_q + S_q' L^H over L'^H L^H.
//
// The column-by-column rule (qr.cu) decides which columns are dependent; this
// path is for matrices without any: it gives up (the flag) as soon as a
// column's part outside the earlier ones is below 1e-4 of the column or 1e-8
// of |A|_F, far above the rule's 1e-10, and the caller runs the column loop
// on the original matrix.  Q and R are then the same as the column loop's up
// to rounding (R has a positive real diagonal, which makes them unique).
//
// Why: 16 M D^2 flops of the column loop take 4.1 ms on the FP64 pipe for a
// 16384 x 128 matrix, and its 128 columns as many grid synchronisations
// (8.5 ms measured); here the rows are read by ~10 launches per panel and
// pass.  Measured, ms per call, column loop (with its rows spread over all SMs)
// and panels: 16384 x 128 7.5 and 1.95, 10368 x 81 2.9 and 1.14, 6561 x 128 4.2
// and 1.5, 4096 x 64 1.25 and 0.67, 81 x 81 1.1 and 0.46.
#include "common.cuh"

#include <algorithm>
#include <cstring>

namespace {

constexpr int PB = QR_PANEL;       // panel width
constexpr int CT = 512;            // threads of the Cholesky kernel
constexpr double MIN_COL2 = 1e-8;  // residual^2 / |column|^2
constexpr double MIN_FRO2 = 1e-16; // residual^2 / |A|_F^2

// G = Sw + Gq (bp x bp, Hermitian; Sw with leading dimension ld, Gq with PB,
// nullptr: none) = L L^H; T = L^-H into rows [n, n + bp) of C (leading
// dimension ld), L^H into Rm (PB x PB).  One block: right-looking Cholesky, the
// same eliminations applied to the identity give L^-1.  pass 2 expects a
// matrix near the identity.  Sets *flag when a pivot is too small.
__global__ void __launch_bounds__(CT) panel_chol_kernel(const cplx* Sw, long long ld, const cplx* Gq, int bp, cplx* C,
                                                        cplx* Rm, const double* fro2, int pass, int* flag) {
    pdl_begin();
    __shared__ cplx G[PB][PB + 1], X[PB][PB + 1];
    __shared__ double norm2[PB], s_inv, s_r;
    __shared__ int bad;
    const int t = threadIdx.x;
    if (*(volatile int*)flag) return;   // an earlier panel gave up
    if (t == 0) bad = 0;
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
            const bool ok = pass == 1 ? (d >= MIN_COL2 * norm2[k] && d > MIN_FRO2 * fro2[0]) : d >= 0.25;
            if (!ok || !isfinite(d)) bad = 1;
            s_inv = rsqrt(d);
            s_r = d * s_inv;
        }
        __syncthreads();
        if (bad) {
            if (t == 0) *flag = 1;
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
                if (t == k) G[k][k].x = s_r;
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
        const int i = e % bp, j = e / bp;   // upper triangular: T = X^H, L^H
        cplx v = make_double2(0.0, 0.0), r = v;
        if (i <= j) {
            v = make_double2(X[j][i].x, -X[j][i].y);
            r = make_double2(G[j][i].x, i == j ? 0.0 : -G[j][i].y);
        }
        C[i + j * ld] = v;
        Rm[i + j * PB] = r;
    }
}

// R's panel (columns n.., leading dimension D): rows < n: S1 + S2 R1, rows
// n .. n + bp: R2 R1.  (S1, S2: leading dimension ld; R1, R2: PB.)
__global__ void panel_r_kernel(const cplx* S1, const cplx* S2, long long ld, const cplx* R1, const cplx* R2, int n,
                               int bp, cplx* R, int D, int* dep, const int* flag, Publish pub) {
    pdl_begin();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e == 0 && pub.hs) {
        pub.hs->qr_flag = *flag;
        if (pub.tc_flag && *(volatile const int*)pub.tc_flag) pub.hs->tc_flag = 1;
        __threadfence_system();
        *(volatile unsigned*)&pub.hs->seq = pub.seq;
    }
    if (e < bp) dep[n + e] = 0;
    if (e >= (n + bp) * bp) return;
    const int i = e % (n + bp), j = e / (n + bp);
    const cplx* L = i < n ? S2 + i : R2 + (i - n);
    const long long s = i < n ? ld : PB;
    cplx a = i < n ? S1[i + j * ld] : make_double2(0.0, 0.0);
    for (int l = i < n ? 0 : i - n; l <= j; ++l) {   // R1 (and R2) upper triangular
        const cplx x = L[l * s], y = R1[l + j * PB];
        a.x = fma(x.x, y.x, fma(-x.y, y.y, a.x));
        a.y = fma(x.x, y.y, fma(x.y, y.x, a.y));
    }
    if (i - n == j) a.y = 0.0;
    R[i + (long long)(n + j) * D] = a;
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

GemmArgs update_args(cplx* A, int M, int n, int bp, const cplx* C) {   // W = [Q W] C, in place
    GemmArgs g = args(M, bp, n + bp);
    g.A = A; g.a_m = 1; g.a_ki = M;
    g.B = C; g.b_ki = 1; g.b_n = n + bp;
    g.C = A + (long long)n * M; g.c_m = 1; g.c_n = M;
    return g;
}

}  // namespace

size_t qr_panel_workspace(int M, int D) {
    size_t need = 0;
    for (int n = 0; n < D; n += PB) {
        const int bp = std::min(PB, D - n);
        need = std::max(need, std::max(digits_workspace_bytes(gram_args(nullptr, M, n, bp, nullptr)),
                                       digits_workspace_bytes(update_args(nullptr, M, n, bp, nullptr))));
    }
    return need;
}

int qr_panel(cplx* A, int M, int D, cplx* R, QrScratch& ws, cudaStream_t s, void* workspace, size_t workspace_bytes,
             int first, int last, const Publish& pub) {
    cplx* S1 = ws.panel;
    cplx* S2 = S1 + (long long)(D + PB) * PB;
    cplx* C = S2 + (long long)(D + PB) * PB;
    cplx* Gq = C + (long long)(D + PB) * PB;
    cplx* R1 = Gq + PB * PB;
    cplx* R2 = R1 + PB * PB;
    int* flag = ws.err + 1;
    int launches = 0;
    for (int n = first; n < std::min(D, last); n += PB) {
        const int bp = std::min(PB, D - n), ld = n + bp;
        for (int pass = 1; pass <= 2; ++pass) {
            cplx* S = pass == 1 ? S1 : S2;
            int l = launch_zgemm_digits(gram_args(A, M, n, bp, S), s, workspace, workspace_bytes);
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
            launch(panel_chol_kernel, 1, CT, 0, s, S + n, ld, n > 0 ? Gq : nullptr, bp, C + n, pass == 1 ? R1 : R2,
                   ws.scal, pass, flag);
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
            l = launch_zgemm_digits(update_args(A, M, n, bp, C), s, workspace, workspace_bytes);
            if (l < 0) return -1;
            launches += l;
        }
        launch(panel_r_kernel, ((n + bp) * bp + 127) / 128, 128, 0, s, S1, S2, ld, R1, R2, n, bp, R, D, ws.flags,
               flag, n + PB >= std::min(D, last) ? pub : Publish{});
        ++launches;
    }
    return launches;
}
