// Truncated SVD of a bond matrix (Sec. "Tensor network simulations": the
// bond dimension chi bounds the kept singular values).  A = Q R by the
// gauge-move QR (qr.cu), then a one-sided (Hestenes) Jacobi SVD of the small
// square factor R = U_R S V^H on the GPU, then U = Q U_R.
//
// Jacobi: columns r_i, r_j of R are rotated until every pair is orthogonal
// to |r_i^H r_j| <= tol ||r_i|| ||r_j||.  One sweep visits every pair once in
// round-robin order (N' - 1 rounds of N'/2 disjoint pairs, N' = N rounded up
// to even); one cooperative launch runs all sweeps, one block per pair of a
// round, with a grid barrier between rounds (pairs whose inner product is
// below 1e-30 |R|_F^2 are treated as orthogonal).  Complex rotation of a pair with
// alpha = |r_i|^2, beta = |r_j|^2, gamma = r_i^H r_j = g e^{i phi}:
//   zeta = (beta - alpha) / (2 g),  t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)),
//   c = 1 / sqrt(1 + t^2),  s = c t,
//   r_i <- c r_i - s e^{-i phi} r_j,   r_j <- s r_i + c e^{-i phi} r_j,
// and the same on the columns of V (so that R_0 V = R stays true); then
// sigma_i = |r_i| and U_R's columns are r_i / sigma_i.
#include "common.cuh"

#include <cmath>

namespace {

constexpr int SVD_THREADS = 128;   // at most; fewer for short columns
constexpr int SVD_ROWS = 2;        // column elements per thread (N <= 256)
constexpr unsigned long long SVD_WAIT_NS = 2000000000ull;   // 2 s per barrier wait

__device__ __forceinline__ unsigned long long svd_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid barrier: arrival counter bar[0], generation bar[1].  Bounded: a wait
// that gives up sets *err and every block leaves at its next barrier.
__device__ bool svd_grid_sync(unsigned* bar, unsigned nblocks, int* err) {
    __syncthreads();
    __shared__ int ok;
    if (threadIdx.x == 0) {
        ok = 1;
        volatile unsigned* vb = bar;
        const unsigned gen = vb[1];
        __threadfence();
        const unsigned arrived = atomicAdd(&bar[0], 1u) + 1u;
        if (arrived == nblocks) {
            bar[0] = 0u;
            __threadfence();
            atomicAdd(&bar[1], 1u);
        } else {
            const unsigned long long t0 = svd_ns();
            for (long long i = 0;; ++i) {
                if (vb[1] != gen) break;
                if (*(volatile int*)err) {
                    ok = 0;
                    break;
                }
                if ((i & 63) == 63 && svd_ns() - t0 > SVD_WAIT_NS) {
                    atomicExch(err, 1);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        if (*(volatile int*)err) ok = 0;
    }
    __syncthreads();
    return ok != 0;
}

__device__ void pair_of(int k, int r, int Np, int& i, int& j) {
    // round-robin: position 0 fixed, positions 1..Np-1 rotate by r
    auto at = [&](int m) { return m == 0 ? 0 : 1 + (m - 1 + r) % (Np - 1); };
    i = at(k);
    j = at(Np - 1 - k);
}

// Several matrices in one launch: a sweep over one matrix is a chain of
// barriers between its N / 2 blocks (4 ms at N = 64, nearly all of it waiting),
// so the bonds of a tree run side by side, each with its own barrier.  A round
// is bound by the FP64 pipe (14 bonds of 64: three blocks per SM) and the
// chain load - sums - rotation - store - barrier.  Measured, 14 bonds of 64 one
// after another -> side by side -> with each element loaded once and the scalar
// work spread over lanes: 64 -> 18.1 -> 14.9 ms; one 64 x 64 11.5 -> 10.4.
struct JacobiBatch {
    JacobiTask t[SVD_BATCH];
    int first[SVD_BATCH + 1];   // first block of each matrix
    int n;
};

// info: [0] sweeps run, [1] unused, [2], [3] rotation counters (alternating sweeps)
__global__ void __launch_bounds__(SVD_THREADS) jacobi_kernel(const __grid_constant__ JacobiBatch jb, int max_sweeps,
                                                            double tol, int* err) {
    __shared__ double red[4][SVD_THREADS / 32];
    __shared__ double rot[4];   // c, s, cos phi, sin phi; rot[0] < 0: skip
    int m = 0;
    while ((int)blockIdx.x >= jb.first[m + 1]) ++m;
    cplx* R = jb.t[m].R;
    cplx* V = jb.t[m].V;
    const int N = jb.t[m].N, Np = N + (N & 1);
    unsigned* bar = jb.t[m].bar;
    int* info = jb.t[m].info;
    const unsigned nb = jb.first[m + 1] - jb.first[m];
    const int k = (int)blockIdx.x - jb.first[m];
    // |R|_F^2, the same in every block (same summation order): pairs whose
    // inner product is below 1e-30 |R|_F^2 are left alone -- columns that
    // rank deficiency has already reduced to rounding noise would otherwise
    // be rotated into denormals and overflow the rotation angle
    __shared__ double s_floor;
    {
        double a = 0.0;
        for (long long e = threadIdx.x; e < (long long)N * N; e += blockDim.x) {
            const cplx x = __ldcg(R + e);
            a += x.x * x.x + x.y * x.y;
        }
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if ((threadIdx.x & 31) == 0) red[0][threadIdx.x >> 5] = a;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int q = 0; q < (int)blockDim.x / 32; ++q) t += red[0][q];
            s_floor = 1e-30 * t;
        }
        __syncthreads();
    }
    const double floor_g = s_floor;
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        int* cnt = &info[2 + (sweep & 1)];
        if (k == 0 && threadIdx.x == 0) *cnt = 0;
        if (!svd_grid_sync(bar, nb, err)) return;
        for (int r = 0; r < Np - 1; ++r) {
            int i, j;
            pair_of(k, r, Np, i, j);
            if (i > j) {
                const int t = i;
                i = j;
                j = t;
            }
            if (j < N) {
                // columns move between blocks from round to round: read them
                // through L2 (__ldcg), never from a stale L1 line; each element
                // once, V's in flight while the rotation is worked out
                const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (int)blockDim.x / 32;
                cplx* ci = R + (long long)i * N;
                cplx* cj = R + (long long)j * N;
                cplx* vi = V + (long long)i * N;
                cplx* vj = V + (long long)j * N;
                cplx x[SVD_ROWS], y[SVD_ROWS], vx[SVD_ROWS], vy[SVD_ROWS];
#pragma unroll
                for (int q = 0; q < SVD_ROWS; ++q) {
                    const int e = threadIdx.x + q * (int)blockDim.x;
                    if (e >= N) continue;
                    x[q] = __ldcg(ci + e);
                    y[q] = __ldcg(cj + e);
                }
#pragma unroll
                for (int q = 0; q < SVD_ROWS; ++q) {
                    const int e = threadIdx.x + q * (int)blockDim.x;
                    if (e >= N) continue;
                    vx[q] = __ldcg(vi + e);
                    vy[q] = __ldcg(vj + e);
                }
                if (32 * w < N) {
                    double a = 0.0, b = 0.0, gr = 0.0, gi = 0.0;
#pragma unroll
                    for (int q = 0; q < SVD_ROWS; ++q) {
                        if (threadIdx.x + q * (int)blockDim.x >= N) continue;
                        a += x[q].x * x[q].x + x[q].y * x[q].y;
                        b += y[q].x * y[q].x + y[q].y * y[q].y;
                        gr += x[q].x * y[q].x + x[q].y * y[q].y;   // conj(x) y
                        gi += x[q].x * y[q].y - x[q].y * y[q].x;
                    }
                    // the four sums share the lanes (six FP64 additions, not twenty):
                    // a ends in lanes 0-7, b 8-15, gr 16-23, gi 24-31
                    const bool up = lane & 16, mid = lane & 8;
                    double k0 = up ? gr : a, k1 = up ? gi : b;
                    k0 += __shfl_xor_sync(0xffffffffu, up ? a : gr, 16);
                    k1 += __shfl_xor_sync(0xffffffffu, up ? b : gi, 16);
                    double v = mid ? k1 : k0;
                    v += __shfl_xor_sync(0xffffffffu, mid ? k0 : k1, 8);
                    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    if ((lane & 7) == 0) red[lane >> 3][w] = v;
                } else if ((lane & 7) == 0) {
                    red[lane >> 3][w] = 0.0;
                }
                __syncthreads();
                if (w == 0) {   // lanes work on different quantities: the FP64 pipe takes a warp at a time
                    double v = 0.0;
                    for (int q = 0; q < nw; ++q) v += red[lane & 3][q];
                    const double A = __shfl_sync(0xffffffffu, v, 0), B = __shfl_sync(0xffffffffu, v, 1),
                                 Gr = __shfl_sync(0xffffffffu, v, 2), Gi = __shfl_sync(0xffffffffu, v, 3);
                    v = sqrt((lane & 1) ? A * B : Gr * Gr + Gi * Gi);
                    const double g = __shfl_sync(0xffffffffu, v, 0), ab = __shfl_sync(0xffffffffu, v, 1);
                    if (g > tol * ab && g > floor_g) {
                        v = (lane == 0 ? B - A : lane == 1 ? Gr : Gi) / (lane == 0 ? 2.0 * g : g);
                        const double zeta = __shfl_sync(0xffffffffu, v, 0);
                        const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                        const double c = 1.0 / sqrt(1.0 + t * t);
                        if (lane == 0) {
                            rot[0] = c;
                            rot[1] = c * t;
                            atomicAdd(cnt, 1);
                        } else if (lane < 3) {
                            rot[lane + 1] = v;
                        }
                    } else if (lane == 0) {
                        rot[0] = -1.0;
                    }
                }
                __syncthreads();
                if (rot[0] >= 0.0) {
                    const double c = rot[0], s = rot[1], pc = rot[2], ps = rot[3];   // e^{-i phi} = pc - i ps
                    auto rotate = [&](const cplx& p, const cplx& q, cplx* pi, cplx* pj) {
                        const cplx yp = make_double2(pc * q.x + ps * q.y, pc * q.y - ps * q.x);   // e^{-i phi} q
                        *pi = make_double2(c * p.x - s * yp.x, c * p.y - s * yp.y);
                        *pj = make_double2(s * p.x + c * yp.x, s * p.y + c * yp.y);
                    };
#pragma unroll
                    for (int q = 0; q < SVD_ROWS; ++q) {
                        const int e = threadIdx.x + q * (int)blockDim.x;
                        if (e >= N) continue;
                        rotate(x[q], y[q], ci + e, cj + e);
                        rotate(vx[q], vy[q], vi + e, vj + e);
                    }
                }
            }
            if (!svd_grid_sync(bar, nb, err)) return;
        }
        if (*(volatile int*)cnt == 0) {
            ++sweep;
            break;
        }
    }
    if (k == 0 && threadIdx.x == 0) info[0] = sweep;
}

// sigma_i = |r_i|; rank order (descending, earlier index first on ties);
// kept count k = min(chi, #{sigma >= eps sigma_max}); discarded weight;
// Ur[:, t] = r_order[t] / sigma (t < k), Vh[t, :] = conj(V[:, order[t]]).
// One block.
__global__ void svd_finish_kernel(const cplx* R, const cplx* V, int N, int chi, double eps, cplx* Ur, cplx* Vh,
                                  double* S, int* kout, double* disc, int* order) {
    pdl_begin();
    extern __shared__ double sig[];
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        double s = 0.0;
        for (int e = 0; e < N; ++e) {
            const cplx x = R[(long long)i * N + e];
            s += x.x * x.x + x.y * x.y;
        }
        sig[i] = sqrt(s);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        int rk = 0;
        for (int j = 0; j < N; ++j)
            if (sig[j] > sig[i] || (sig[j] == sig[i] && j < i)) ++rk;
        order[rk] = i;
    }
    __syncthreads();
    __shared__ int k;
    __shared__ double smax, tot, kept;
    if (threadIdx.x == 0) {
        smax = sig[order[0]];
        int n = 0;
        if (eps < 0.0) {   // keep exactly min(chi, N) columns, zero values included
            n = chi < N ? chi : N;
        } else {
            while (n < N && n < chi && sig[order[n]] >= eps * smax && sig[order[n]] > 0.0) ++n;
        }
        if (n == 0) n = 1;
        k = n;
        tot = 0.0;
        kept = 0.0;
        for (int t = 0; t < N; ++t) {
            const double s2 = sig[order[t]] * sig[order[t]];
            tot += s2;
            if (t < n) kept += s2;
        }
        *kout = n;
        *disc = tot > 0.0 ? (tot - kept) / tot : 0.0;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < k; t += blockDim.x) S[t] = sig[order[t]];
    for (long long e = threadIdx.x; e < (long long)N * k; e += blockDim.x) {
        const int t = (int)(e / N), row = (int)(e % N);
        const int i = order[t];
        const double inv = sig[i] > 0.0 ? 1.0 / sig[i] : 0.0;
        const cplx x = R[(long long)i * N + row];
        Ur[e] = make_double2(x.x * inv, x.y * inv);
        const cplx v = V[(long long)i * N + row];
        Vh[t + (long long)k * row] = make_double2(v.x, -v.y);   // Vh is k x N, column-major
    }
}

__global__ void identity_kernel(cplx* V, int N) {
    pdl_begin();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)N * N;
         e += (long long)gridDim.x * blockDim.x)
        V[e] = make_double2((e % N) == (e / N) ? 1.0 : 0.0, 0.0);
}

}  // namespace

int svd_jacobi_batch(const JacobiTask* tasks, int n, int max_sweeps, double tol, int* err, cudaStream_t s) {
    int dev = 0, nsm = 0, per_sm = 0, launches = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int T = 32;   // a thread per column element; idle warps would still take their turns at the FP64 pipe
    for (int i = 0; i < n; ++i) {
        if (tasks[i].N > SVD_ROWS * SVD_THREADS) return -1;
        T = std::max(T, std::min(SVD_THREADS, (tasks[i].N + 31) / 32 * 32));
    }
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_kernel, T, 0);
    const int room = nsm * per_sm;
    for (int i = 0; i < n;) {
        JacobiBatch jb;
        jb.n = 0;
        jb.first[0] = 0;
        for (; i < n && jb.n < SVD_BATCH; ++i) {   // as many matrices as are co-resident
            const JacobiTask& t = tasks[i];
            const int blocks = (t.N + 1) / 2;
            if (jb.n > 0 && jb.first[jb.n] + blocks > room) break;
            launch(identity_kernel, (t.N * t.N + 255) / 256, 256, 0, s, t.V, t.N);
            cudaMemsetAsync(t.bar, 0, 2 * sizeof(unsigned), s);
            cudaMemsetAsync(t.info, 0, 4 * sizeof(int), s);
            ++launches;
            if (t.N < 2) continue;   // nothing to rotate
            jb.t[jb.n] = t;
            jb.first[jb.n + 1] = jb.first[jb.n] + blocks;
            ++jb.n;
        }
        if (jb.n == 0) continue;
        void* args[] = {(void*)&jb, (void*)&max_sweeps, (void*)&tol, (void*)&err};
        if (cudaLaunchCooperativeKernel((const void*)jacobi_kernel, dim3(jb.first[jb.n]), dim3(T), args, 0,
                                        s) != cudaSuccess)
            return -1;
        ++launches;
    }
    return launches;
}

int svd_jacobi_square(cplx* R, cplx* V, int N, int max_sweeps, double tol, unsigned* bar, int* err, int* info,
                      cudaStream_t s) {
    const JacobiTask t{R, V, N, bar, info};
    return svd_jacobi_batch(&t, 1, max_sweeps, tol, err, s);
}

int svd_finish(const cplx* R, const cplx* V, int N, int chi, double eps, cplx* Ur, cplx* Vh, double* S, int* k,
               double* disc, int* order, cudaStream_t s) {
    launch(svd_finish_kernel, 1, 256, sizeof(double) * N, s, R, V, N, chi, eps, Ur, Vh, S, k, disc, order);
    return 1;
}
