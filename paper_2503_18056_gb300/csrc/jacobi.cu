// Small dense factorisations of the Gram-SVD rounding (App. A.2 of arXiv
// 2503.18056) and the rank decision of App. A (note on rank truncation).
//
// 1. Symmetric eigensolver: two-sided cyclic Jacobi with the parallel
//    round-robin ("circle") ordering.  Each round applies n/2 disjoint plane
//    rotations at once: G <- J^T G J, Vt <- J^T Vt.  A CTA owns a few row pairs
//    (p, q) per round: it forms those pairs' rotation angles and publishes them,
//    loads the rows with coalesced L2 reads and rotates them on the left by
//    their own J_k; after a grid-wide barrier it reads every pair's angles,
//    rotates the non-identity column pairs in shared memory and writes the rows
//    to the other buffer (the matrix is double-buffered; a second barrier ends
//    the round).  The three entries (g_pp, g_qq, g_pq) that define the next
//    round's rotations are written by the row owners into a compact array, so
//    the owning CTA reads them with one coalesced load.  Rotation
//    angles follow Golub & Van Loan, Alg. 8.4.1 (symSchur2); a rotation is
//    skipped when |g_pq| <= tol_rel sqrt(|g_pp g_qq|) or |g_pq| <= tol_abs, and
//    the sweeps stop after one that skipped every rotation.
// 2. Pivoted Cholesky of a positive semidefinite matrix, G = W^T W with W
//    upper-trapezoidal in pivot order (left-looking, diagonal pivoting, stopped
//    when the largest remaining diagonal entry is at eps_mach max(diag G)).  The rounding
//    needs from G_B only a factor with W^T W = G_B, which this gives in n
//    sequential steps instead of an eigendecomposition.
//
// Both kernels are persistent: a cooperative launch guarantees co-residency and
// the grid barrier is a bounded spin that latches DEV_TIMEOUT in the status
// word instead of waiting forever.
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include <cooperative_groups.h>

#include "internal.h"
#include "intfp.h"

namespace ttsn {

namespace {

constexpr int JT = 256;
constexpr int MAX_SWEEPS = JACOBI_MAX_SWEEPS;
// control block (ints): [0] barrier arrivals, [1] unused, [2] sweeps,
// [3] pivoted-Cholesky rank, [4 .. 4+MAX_SWEEPS) rotations applied per sweep
constexpr int CTRL_INTS = 8 + MAX_SWEEPS;
constexpr long long SPIN_LIMIT = 1LL << 21;  // ~1 s (an L2 acquire load plus a 32 ns sleep per try)
constexpr int MAX_PAIRS_PER_CTA = 8;

__device__ __forceinline__ void round_pair(int N, int r, int k, int& p, int& q) {
    const int m = N - 1;
    if (k == 0) {
        p = m;
        q = r;
    } else {  // (r + k) mod m and (r - k) mod m for 0 <= r < m, 0 < k < m
        p = r + k;
        if (p >= m) p -= m;
        q = r - k;
        if (q < 0) q += m;
    }
    if (p > q) {
        const int t = p;
        p = q;
        q = t;
    }
}

// Pair index and partner of index x in round r (inverse of round_pair).
__device__ __forceinline__ void pair_of(int N, int r, int x, int& k, int& partner) {
    const int m = N - 1;
    if (x == m) {
        k = 0;
        partner = r;
        return;
    }
    if (x == r) {
        k = 0;
        partner = m;
        return;
    }
    const int d = (x - r + m) % m;  // 1 .. m-1
    if (d <= N / 2 - 1) {
        k = d;
        partner = (r - d + m) % m;
    } else {
        k = m - d;
        partner = (r + k) % m;
    }
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid-wide barrier with a bounded wait.  ctrl[0] counts arrivals over the
// whole launch (the control block is zeroed before every launch), so the
// barrier that a CTA enters for the e-th time completes when the count
// reaches e * nblocks: one release-atomic arrival per CTA, acquire-load
// polling, no reset and no second word to bump.  Returns false (and latches
// DEV_TIMEOUT) if the wait ran out; the other CTAs then never see the count
// complete and run out in turn.  epoch is the caller's barrier counter (its
// value matters in thread 0 only).
__device__ bool grid_barrier(int* ctrl, int* status, unsigned nblocks, unsigned& epoch) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        ++epoch;
        if (nblocks > 1) {
            unsigned* count = reinterpret_cast<unsigned*>(ctrl);
            const unsigned target = epoch * nblocks;
            // the CTA's writes (every thread's, ordered by the __syncthreads
            // above) become visible GPU-wide before the arrival is counted
            __threadfence();
            const unsigned old = atomicAdd(count, 1u);
            if (old + 1u < target) {
                long long it = 0;
                while (ld_acquire(count) < target) {
                    if (++it > SPIN_LIMIT) {
                        ok = 0;
                        atomicOr(status, DEV_TIMEOUT);
                        break;
                    }
                    __nanosleep(32);
                }
            }
            __threadfence();
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

__global__ void jacobi_init_kernel(int n, int N, const double* __restrict__ G, long ldg, double* g0,
                                   double* vt, long ld, double* abc, const int* n_dev) {
    if (n_dev) {
        n = *n_dev;
        N = n + (n & 1);
        ldg = ld = n;
    }
    const long total = (long)n * n;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int i = (int)(t / n), j = (int)(t % n);
        g0[(long)i * ld + j] = G[(long)i * ldg + j];
        vt[(long)i * ld + j] = (i == j) ? 1.0 : 0.0;
    }
    // entries of the round-0 pairs
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < N / 2; k += gridDim.x * blockDim.x) {
        int p, q;
        round_pair(N, 0, k, p, q);
        if (q < n) {
            abc[3 * k] = G[(long)p * ldg + p];
            abc[3 * k + 1] = G[(long)q * ldg + q];
            abc[3 * k + 2] = 0.5 * (G[(long)p * ldg + q] + G[(long)q * ldg + p]);
        } else {
            abc[3 * k] = abc[3 * k + 1] = abc[3 * k + 2] = 0.0;
        }
    }
}

// One launch runs every sweep.  A round has two grid barriers:
//  A. each CTA forms the rotation angles of the pairs it owns only (from the
//     compact entries the previous round published), publishes them, and
//     left-rotates its own row pairs and eigenvector rows;
//  B. after the barrier every CTA reads all angles with one coalesced load,
//     compacts the list of pairs whose rotation is not the identity, applies
//     those column rotations to its own rows, stores the rows to the other
//     buffer and publishes the next round's pair entries.
// Forming each angle once instead of once per CTA is what the second barrier
// buys: on GB300 a CTA that formed all n/2 angles itself spent about as long
// on their FP64 square roots and divisions as on the rotations, and skipped
// (identity) rotations cost nothing in the later sweeps.
__global__ void __launch_bounds__(JT)
jacobi_kernel(int n, int N, double* g0, double* g1, long ld, double* vt, double* abc0,
              double* abc1, double* cs_g, double* lam_out, int* ctrl, int* status, double tol_rel,
              double tol_abs_rel, int max_sweeps, const int* n_dev) {
    if (n_dev) {  // a captured step: the grid and shared memory fit the largest n
        n = *n_dev;
        N = n + (n & 1);
        ld = n;
    }
    extern __shared__ double sm[];
    const int npairs = N / 2;
    // pairs this CTA owns: k = blockIdx.x + i * gridDim.x < npairs
    const int mine = max(0, (npairs - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x);
    double* cs = sm;                                     // 2 * npairs: c, s of every pair
    double* rows = cs + 2 * npairs;                      // 2 * ppc rows of n
    int* act = reinterpret_cast<int*>(rows + 2 * (size_t)((npairs + gridDim.x - 1) / gridDim.x) * n);
    __shared__ int s_cnt;
    __shared__ int s_done;
    __shared__ int s_nact;
    __shared__ int s_wsum[JT / 32];
    __shared__ double s_dmax;

    unsigned epoch = 0;
    double* cur = g0;
    double* nxt = g1;
    double* abc_cur = abc0;
    double* abc_nxt = abc1;
    if (threadIdx.x == 0) {
        double dm = 0.0;
        for (int i = 0; i < n; ++i) dm = fmax(dm, fabs(__ldcg(g0 + (long)i * ld + i)));
        s_dmax = dm;
    }
    __syncthreads();
    const double tol_abs = tol_abs_rel * s_dmax;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        if (threadIdx.x == 0) s_cnt = 0;
        __syncthreads();
        for (int r = 0; r < N - 1; ++r) {
            const int rn = (r + 1 == N - 1) ? 0 : r + 1;  // next round (wraps to the next sweep)
            // A1. the angles of the owned pairs (Golub & Van Loan, Alg. 8.4.1)
            if (threadIdx.x < mine) {
                const int i = threadIdx.x;
                const int k = blockIdx.x + i * gridDim.x;
                int p, q;
                round_pair(N, r, k, p, q);
                double c = 1.0, s = 0.0;
                if (q < n) {
                    const double a = __ldcg(abc_cur + 3 * k);
                    const double b = __ldcg(abc_cur + 3 * k + 1);
                    const double o = __ldcg(abc_cur + 3 * k + 2);
                    const double ao = fabs(o);
                    if (ao > tol_abs && ao > tol_rel * sqrt(fabs(a) * fabs(b))) {
                        const double tau = (b - a) / (2.0 * o);
                        const double t =
                            (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
                        c = 1.0 / sqrt(1.0 + t * t);
                        s = t * c;
                        atomicAdd(&s_cnt, 1);
                    }
                }
                cs[2 * k] = c;
                cs[2 * k + 1] = s;
                __stcg(cs_g + 2 * k, c);
                __stcg(cs_g + 2 * k + 1, s);
            }
            __syncthreads();
            // A2. load and left-rotate every owned row pair; rotate its eigenvector rows
            for (int i = 0; i < mine; ++i) {
                const int k = blockIdx.x + i * gridDim.x;
                int p, q;
                round_pair(N, r, k, p, q);
                const bool hp = p < n, hq = q < n;
                const double c = cs[2 * k], s = cs[2 * k + 1];
                double* rp = rows + (2 * i) * n;
                double* rq = rp + n;
                if (s != 0.0) {
#pragma unroll 4
                    for (int j = threadIdx.x; j < n; j += blockDim.x) {
                        const double xp = __ldcg(cur + (long)p * ld + j);
                        const double xq = __ldcg(cur + (long)q * ld + j);
                        rp[j] = c * xp - s * xq;
                        rq[j] = s * xp + c * xq;
                        const double vp = __ldcg(vt + (long)p * ld + j);
                        const double vq = __ldcg(vt + (long)q * ld + j);
                        __stcg(vt + (long)p * ld + j, c * vp - s * vq);
                        __stcg(vt + (long)q * ld + j, s * vp + c * vq);
                    }
                } else {
#pragma unroll 4
                    for (int j = threadIdx.x; j < n; j += blockDim.x) {
                        rp[j] = hp ? __ldcg(cur + (long)p * ld + j) : 0.0;
                        rq[j] = hq ? __ldcg(cur + (long)q * ld + j) : 0.0;
                    }
                }
            }
            if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return;
            // B1. every pair's angles, and the list of the non-identity ones
            for (int k = threadIdx.x; k < npairs; k += blockDim.x) {
                cs[2 * k] = __ldcg(cs_g + 2 * k);
                cs[2 * k + 1] = __ldcg(cs_g + 2 * k + 1);
            }
            __syncthreads();
            {
                // block-wide compaction in pair order: chunks of blockDim.x pairs
                int base = 0;
                for (int k0 = 0; k0 < npairs; k0 += blockDim.x) {
                    const int k = k0 + threadIdx.x;
                    const bool on = k < npairs && cs[2 * k + 1] != 0.0;
                    const unsigned bal = __ballot_sync(0xffffffffu, on);
                    if (lane == 0) s_wsum[warp] = __popc(bal);
                    __syncthreads();
                    int before = 0, total = 0;
                    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
                        if (w < warp) before += s_wsum[w];
                        total += s_wsum[w];
                    }
                    if (on) act[base + before + __popc(bal & ((1u << lane) - 1u))] = k;
                    base += total;
                    __syncthreads();
                }
                if (threadIdx.x == 0) s_nact = base;
            }
            __syncthreads();
            const int nact = s_nact;
            // B2. right rotations of the non-identity column pairs, on all owned rows
            const int nrows = 2 * mine;
            for (int a = threadIdx.x; a < nact; a += blockDim.x) {
                const int kk = act[a];
                int pp, qq;
                round_pair(N, r, kk, pp, qq);
                const double c2 = cs[2 * kk], s2 = cs[2 * kk + 1];
                for (int row = 0; row < nrows; ++row) {
                    double* rr = rows + row * n;
                    const double a0 = rr[pp], b0 = rr[qq];
                    rr[pp] = c2 * a0 - s2 * b0;
                    rr[qq] = s2 * a0 + c2 * b0;
                }
            }
            __syncthreads();
            // B3. exact zeros for the rotated pairs
            if (threadIdx.x < mine) {
                const int i = threadIdx.x;
                const int k = blockIdx.x + i * gridDim.x;
                int p, q;
                round_pair(N, r, k, p, q);
                if (q < n && cs[2 * k + 1] != 0.0) {
                    rows[(2 * i) * n + q] = 0.0;
                    rows[(2 * i + 1) * n + p] = 0.0;
                }
            }
            __syncthreads();
            // B4. store rows and publish the next round's entries
            for (int i = 0; i < mine; ++i) {
                const int k = blockIdx.x + i * gridDim.x;
                int p, q;
                round_pair(N, r, k, p, q);
                const bool hp = p < n, hq = q < n;
                const double* rp = rows + (2 * i) * n;
                const double* rq = rp + n;
                for (int j = threadIdx.x; j < n; j += blockDim.x) {
                    if (hp) __stcg(nxt + (long)p * ld + j, rp[j]);
                    if (hq) __stcg(nxt + (long)q * ld + j, rq[j]);
                }
                if (threadIdx.x < 2) {
                    const int x = threadIdx.x == 0 ? p : q;
                    const double* rx = threadIdx.x == 0 ? rp : rq;
                    if (x < n) {
                        int k2, partner;
                        pair_of(N, rn, x, k2, partner);
                        if (partner < n) {
                            if (x < partner) {
                                __stcg(abc_nxt + 3 * k2, rx[x]);
                                __stcg(abc_nxt + 3 * k2 + 2, rx[partner]);
                            } else {
                                __stcg(abc_nxt + 3 * k2 + 1, rx[x]);
                            }
                        }
                    }
                }
            }
            if (r == N - 2 && threadIdx.x == 0) atomicAdd(ctrl + 4 + sweep, s_cnt);
            if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return;
            double* t = cur;
            cur = nxt;
            nxt = t;
            t = abc_cur;
            abc_cur = abc_nxt;
            abc_nxt = t;
        }
        if (threadIdx.x == 0) s_done = (atomicAdd(ctrl + 4 + sweep, 0) == 0);
        __syncthreads();
        if (s_done) break;
    }
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) {
            ctrl[2] = min(sweep + 1, max_sweeps);
            if (sweep >= max_sweeps) atomicOr(status, DEV_NOT_CONVERGED);
        }
        // eigenvalues: the diagonal of the last written buffer
        for (int i = threadIdx.x; i < n; i += blockDim.x) lam_out[i] = __ldcg(cur + (long)i * ld + i);
    }
}

// One-sided Jacobi on the rows of a factor W (k x n, ld n) with W^T W = K
// (Demmel & Veselic, SIAM J. Matrix Anal. Appl. 13, 1992: the eigenpairs of a
// positive definite matrix from its Cholesky factor by one-sided Jacobi, as
// accurate as two-sided Jacobi on K).  Row pairs follow the same round-robin
// ordering; one warp owns a pair for the round: it forms c = w_p . w_q, and
// if |c| > tol sqrt(a b) (a, b the squared row norms, kept in nrm) rotates the
// two rows so that they become orthogonal and recomputes their norms from the
// rotated rows.  A rotation touches only its own two rows, so a round needs
// one grid barrier and no exchange of angles.  On convergence the rows are
// orthogonal: K = sum_i w_i w_i^T, eigenvalue ||w_i||^2, eigenvector
// w_i / ||w_i||; rows k .. n-1 (K's null space below the factor's floor)
// get eigenvalue 0 and a zero vector.  A negative rank (the factorisation met
// Inf or NaN) gives NaN eigenvalues, which the rank decision reports.
constexpr int OSJ_MAX_WARPS = 8;
constexpr int OSJ_CLUSTER_N = 256;  // sizes solved on one thread-block cluster

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One pair of rows of any length, streamed from L2: c = w_p . w_q, the rotation
// if it is needed, the rotated rows' norms.  Returns whether it rotated.
__device__ __forceinline__ bool osj_pair(double* wp, double* wq, int n, int lane, double* nrm_p, double* nrm_q,
                                         double tol) {
    double c0 = 0.0, c1 = 0.0;
    {
        int j = lane;
        for (; j + 32 < n; j += 64) {
            c0 = fma(__ldcg(wp + j), __ldcg(wq + j), c0);
            c1 = fma(__ldcg(wp + j + 32), __ldcg(wq + j + 32), c1);
        }
        if (j < n) c0 = fma(__ldcg(wp + j), __ldcg(wq + j), c0);
    }
    const double c = warp_sum(c0 + c1);
    const double a = __ldcg(nrm_p), b = __ldcg(nrm_q);
    if (!(a > 0.0 && b > 0.0 && fabs(c) > tol * sqrt(a * b))) return false;
    // Golub & Van Loan, Alg. 8.4.1 on [[a, c], [c, b]]
    const double tau = (b - a) / (2.0 * c);
    const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
    const double cs = 1.0 / sqrt(1.0 + t * t);
    const double sn = t * cs;
    // the rotation moves t c from one squared norm to the other: the growing
    // one is updated by that sum (no cancellation), the shrinking one is
    // summed again from the rotated row
    const bool p_shrinks = t * c > 0.0;
    double ns = 0.0;
    for (int j = lane; j < n; j += 32) {
        const double xo = __ldcg(wp + j), yo = __ldcg(wq + j);
        const double xn = cs * xo - sn * yo;
        const double yn = sn * xo + cs * yo;
        __stcg(wp + j, xn);
        __stcg(wq + j, yn);
        const double v = p_shrinks ? xn : yn;
        ns = fma(v, v, ns);
    }
    ns = warp_sum(ns);
    if (lane == 0) {
        __stcg(nrm_p, p_shrinks ? ns : a - t * c);
        __stcg(nrm_q, p_shrinks ? b + t * c : ns);
    }
    return true;
}

// Squared norms of rows 0 .. k-1, summed from the rows (one warp per row).
__device__ __forceinline__ void osj_norms(const double* W, int n, int k, double* nrm, int gw, int nw, int lane) {
    for (int i = gw; i < k; i += nw) {
        const double* wi = W + (long)i * n;
        double a = 0.0;
        for (int j = lane; j < n; j += 32) {
            const double v = __ldcg(wi + j);
            a = fma(v, v, a);
        }
        a = warp_sum(a);
        if (lane == 0) __stcg(nrm + i, a);
    }
}

__global__ void __launch_bounds__(32 * OSJ_MAX_WARPS)
osj_kernel(int n, const int* __restrict__ k_dev, double* W, double* nrm, double* lam_u, double* vt_u, int* ctrl,
           int* status, int max_sweeps, const int* n_dev, int nsmall) {
    if (n_dev) {  // a captured step: sizes up to nsmall take the launches before it
        n = *n_dev;
        if (n <= nsmall) return;  // every CTA, before any barrier
    }
    // relative skip threshold sqrt(n) eps_mach, the one of LAPACK's one-sided
    // Jacobi SVD (dgesvj): the typical rounding error of a computed inner
    // product of length n, so rounding noise does not keep pairs rotating
    const double tol = sqrt((double)n) * 2.220446049250313e-16;
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const int gw = blockIdx.x * wpb + (threadIdx.x >> 5);
    const int nw = gridDim.x * wpb;
    const int kraw = *k_dev;
    if (kraw < 0) {  // every CTA returns before any barrier
        for (int i = gw; i < n; i += nw) {
            if (lane == 0) lam_u[i] = __longlong_as_double(0x7ff8000000000000LL);
            for (int j = lane; j < n; j += 32) vt_u[(long)i * n + j] = 0.0;
        }
        return;
    }
    const int k = min(kraw, n);
    unsigned epoch = 0;
    __shared__ int s_cnt;
    __shared__ int s_done;
    const int N = k + (k & 1), npairs = N / 2;
    int sweep = 0;
    if (k >= 2) {
        for (; sweep < max_sweeps; ++sweep) {
            if (threadIdx.x == 0) s_cnt = 0;
            // norms summed afresh at every sweep: the updates inside a sweep
            // only steer the angles and the skip test
            osj_norms(W, n, k, nrm, gw, nw, lane);
            if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return;
            int mine = 0;
            for (int r = 0; r < N - 1; ++r) {
                for (int kk = gw; kk < npairs; kk += nw) {
                    int p, q;
                    round_pair(N, r, kk, p, q);
                    if (q >= k) continue;
                    if (osj_pair(W + (long)p * n, W + (long)q * n, n, lane, nrm + p, nrm + q, tol)) ++mine;
                }
                if (r == N - 2) {
                    if (lane == 0 && mine) atomicAdd(&s_cnt, mine);
                    __syncthreads();
                    if (threadIdx.x == 0) atomicAdd(ctrl + 4 + sweep, s_cnt);
                }
                if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return;
            }
            if (threadIdx.x == 0) s_done = (atomicAdd(ctrl + 4 + sweep, 0) == 0);
            __syncthreads();
            if (s_done) break;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctrl[2] = k >= 2 ? min(sweep + 1, max_sweeps) : 0;
        if (k >= 2 && sweep >= max_sweeps) atomicOr(status, DEV_NOT_CONVERGED);
    }
    // eigenvalues: the converged rows' squared norms, summed from the rows
    osj_norms(W, n, k, nrm, gw, nw, lane);
    if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return;
    for (int i = gw; i < n; i += nw) {
        const double a = i < k ? __ldcg(nrm + i) : 0.0;
        const double f = a > 0.0 ? 1.0 / sqrt(a) : 0.0;
        if (lane == 0) lam_u[i] = a;
        const double* wi = W + (long)i * n;
        for (int j = lane; j < n; j += 32) vt_u[(long)i * n + j] = i < k ? f * __ldcg(wi + j) : 0.0;
    }
}

// Up to OSJ_CLUSTER_N rows on one thread-block cluster: osj_kernel's rotations in
// the same order, laid out for what bounds it on GB300, FP64 issue (64 clocks a warp
// instruction and SM sub-partition, about 600 for a square root or a division)
// and the latency of a round:
// - The rows never leave the SMs.  A warp holds a pair's rows in registers and
//   after the round sends each into the shared memory of the warp that needs it
//   next: two short remote stores and one hardware cluster barrier a round, no
//   trip to L2.  The pairs are round_pair's: slot 0 holds the last row, which
//   stays, and row r; slot k rows r + k (first) and r - k (second); from round to
//   round the first rows move down a slot, the second rows up one, and the ends
//   turn.  (Two pairs a warp above 128 rows, half the FP64 instructions of the
//   angle a sub-partition: 7.2 ms against 6.2 at n = 163, equal at 241 to 256.)
// - The angle's quotients and roots are intfp.h's, the same bits from integer
//   instructions (n = 61: 1.76 -> 1.40 ms, 163: 8.0 -> 6.2).
// - A rotated row's squared norm is summed over the lanes by the warp that takes
//   it next, together with that warp's inner product: six shuffle-and-add steps
//   for three sums, where one sum alone takes five.
// - The skip test compares exponents and forms tol sqrt(a b) only within a few
//   binades of it; an angle with |tau| >= 2^28 needs neither square root, where
//   sqrt(1 + tau^2) = |tau| and sqrt(1 + t^2) = 1 exactly (the two roundings stay
//   within half an ulp of tau: relative errors 2^-54 / m^2 + 2^-57 against 2^-53 /
//   m for a significand m below sqrt 2, 2^-53 / m^2 + 2^-57 above).
// Measured (GB300, factorisation included, a graded full-rank matrix): n = 61
// 2.9 -> 1.40 ms, 128 6.4 -> 3.3, 163 11.1 -> 6.2, 256 22.9 -> 14.5.
// inbox: [slot of this CTA][parity][first, second][32 (C + 1)], a row's entries
// and its norm's partial sums, then the rows' squared norms and indices.
struct OsjMeta {
    double nrm;
    int idx, part;  // part: the squared norm follows from the row's partial sums
};

// 2 log2|c| against log2(tol^2 a b): +1 certainly above, -1 certainly below, 0 close
__device__ __forceinline__ int osj_far(double c, double a, double b, double tol) {
    auto ex = [](double v) { return (int)((__double2hiint(v) >> 20) & 0x7FF); };
    const int ec = ex(c), ea = ex(a), eb = ex(b), et = ex(tol);
    if (ec == 0 || ea == 0 || eb == 0 || ec == 0x7FF || ea == 0x7FF || eb == 0x7FF) return 0;
    // c^2 in [2^(2 ec), 2^(2 ec + 2)), tol^2 a b in [2^s, 2^(s + 4)) (biases: 2 and 4)
    const int s = 2 * et + ea + eb - 2 * 1023;
    if (abs(ea + eb - 2 * 1023) > 1000) return 0;  // a b near the range's ends
    return 2 * ec >= s + 5 ? 1 : (2 * ec + 2 <= s - 1 ? -1 : 0);
}

// 2 v, without the FP64 pipe
__device__ __forceinline__ double twice(double v) {
    const int hi = __double2hiint(v), ex = (hi >> 20) & 0x7FF;
    return (unsigned)(ex - 1) < 0x7FDu ? __hiloint2double(hi + (1 << 20), __double2loint(v)) : v + v;
}

// tan, cos and sin of the rotation that makes [[a, c], [c, b]] diagonal (Golub &
// Van Loan, Alg. 8.4.1), c far from 0
__device__ __forceinline__ void osj_angle(double a, double b, double c, double& t, double& cs, double& sn) {
    const double tau = intfp::div(b - a, twice(c));
    const double at = fabs(tau);
    if (at >= 268435456.0 && at < 1e150) {
        t = intfp::div(tau >= 0.0 ? 1.0 : -1.0, twice(at));
        cs = 1.0;
        sn = t;
    } else {
        t = intfp::div(tau >= 0.0 ? 1.0 : -1.0, at + intfp::root(1.0 + tau * tau));
        cs = intfp::div(1.0, intfp::root(1.0 + t * t));
        sn = t * cs;
    }
}

// Three sums over a warp at once: a group of lanes carries a different one from
// each step on, every sum with the additions of its own butterfly.
__device__ __forceinline__ void osj_sum3(double& c, double& px, double& py, int lane) {
    const bool h1 = lane & 16, h2 = lane & 8;
    double u = (h1 ? px : c) + __shfl_xor_sync(0xffffffffu, h1 ? c : px, 16);
    const double v = py + __shfl_xor_sync(0xffffffffu, py, 16);
    u = (h2 ? v : u) + __shfl_xor_sync(0xffffffffu, h2 ? u : v, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    c = __shfl_sync(0xffffffffu, u, 0);
    py = __shfl_sync(0xffffffffu, u, 8);
    px = __shfl_sync(0xffffffffu, u, 16);
}

template <int C>
__device__ void osj_cluster_body(int n, int k, const double* W, double* lam_u, double* vt_u, int* ctrl, int* status,
                                 int max_sweeps, double tol, double* inbox) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int ROW = 32 * (C + 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int slot = blockIdx.x * wpb + warp;
    const int N = k + (k & 1), S = N / 2;
    const bool active = slot < S;
    OsjMeta* meta = reinterpret_cast<OsjMeta*>(inbox + (size_t)wpb * 4 * ROW);
    double x[C], y[C];
    auto norm2 = [&](const double (&v)[C]) {
        double p = 0.0;
#pragma unroll
        for (int e = 0; e < C; ++e) p = fma(v[e], v[e], p);
        return warp_sum(p);
    };
    // x: the row of the smaller index; sw: it is the slot's second row
    int ix = 0, iy = 0;
    bool sw = false;
    double a = 0.0, b = 0.0;    // squared norms; pa, pb: their partial sums where fa, fb
    double pa = 0.0, pb = 0.0;
    bool fa = false, fb = false;
    {
        const int i0 = slot == 0 ? N - 1 : slot, i1 = slot == 0 ? 0 : N - 1 - slot;  // round 0
        sw = i1 < i0;
        ix = min(i0, i1);
        iy = max(i0, i1);
#pragma unroll
        for (int e = 0; e < C; ++e) {
            const int j = lane + 32 * e;
            x[e] = active && ix < k && j < n ? __ldcg(W + (long)ix * n + j) : 0.0;
            y[e] = active && iy < k && j < n ? __ldcg(W + (long)iy * n + j) : 0.0;
        }
    }
    // where the slot's rows go after a round
    double *to0 = nullptr, *to1 = nullptr;
    OsjMeta *me0 = nullptr, *me1 = nullptr;
    if (active && S > 1) {
        const int ds0 = slot == 0 ? 0 : slot - 1, dw0 = slot == 1 ? 1 : 0;
        const int ds1 = slot == S - 1 ? slot : slot + 1, dw1 = slot != 0 && slot == S - 1 ? 0 : 1;
        to0 = cl.map_shared_rank(inbox, ds0 / wpb) + ((size_t)(ds0 % wpb) * 4 + dw0) * ROW;
        to1 = cl.map_shared_rank(inbox, ds1 / wpb) + ((size_t)(ds1 % wpb) * 4 + dw1) * ROW;
        me0 = cl.map_shared_rank(meta, ds0 / wpb) + (ds0 % wpb) * 4 + dw0;
        me1 = cl.map_shared_rank(meta, ds1 / wpb) + (ds1 % wpb) * 4 + dw1;
    }
    cl.sync();  // every CTA of the cluster runs before its shared memory is written
    int sweep = 0;
    bool done = k < 2;
    for (; sweep < max_sweeps && !done; ++sweep) {
        // norms summed afresh at every sweep: the updates inside a sweep only
        // steer the angles and the skip test
        a = norm2(x);
        b = norm2(y);
        fa = fb = false;
        int mine = 0;
        for (int r = 0; r < N - 1; ++r) {
            const int par = r & 1;
            {
                double c0 = 0.0, c1 = 0.0;
#pragma unroll
                for (int e = 0; e < C; ++e) {
                    if (e & 1)
                        c1 = fma(x[e], y[e], c1);
                    else
                        c0 = fma(x[e], y[e], c0);
                }
                double c = C == 1 ? c0 : c0 + c1;
                if (fa || fb) {
                    osj_sum3(c, pa, pb, lane);
                    a = fa ? pa : a;
                    b = fb ? pb : b;
                    fa = fb = false;
                } else {
                    c = warp_sum(c);
                }
                bool rot = false;
                if (active && iy < k && a > 0.0 && b > 0.0) {
                    const int far = osj_far(c, a, b, tol);
                    rot = far > 0 || (far == 0 && fabs(c) > tol * sqrt(a * b));
                }
                if (rot) {
                    double t, cs, sn;
                    osj_angle(a, b, c, t, cs, sn);
                    // the rotation moves t c from one squared norm to the other: the
                    // growing one is updated by that sum (no cancellation), the
                    // shrinking one is summed again from the rotated row, over the
                    // lanes with the next product
                    const bool p_shrinks = t * c > 0.0;
                    double ns = 0.0;
#pragma unroll
                    for (int e = 0; e < C; ++e) {
                        const double xn = cs * x[e] - sn * y[e];
                        const double yn = sn * x[e] + cs * y[e];
                        x[e] = xn;
                        y[e] = yn;
                        const double v = p_shrinks ? xn : yn;
                        ns = fma(v, v, ns);
                    }
                    if (p_shrinks) {
                        b = b + t * c;
                        pa = ns;
                    } else {
                        a = a - t * c;
                        pb = ns;
                    }
                    fa = p_shrinks;
                    fb = !p_shrinks;
                    ++mine;
                }
            }
            if (active && S > 1) {
                double *o0 = (sw ? to1 : to0) + par * 2 * ROW, *o1 = (sw ? to0 : to1) + par * 2 * ROW;
#pragma unroll
                for (int e = 0; e < C; ++e) {
                    o0[lane + 32 * e] = x[e];
                    o1[lane + 32 * e] = y[e];
                }
                if (fa) o0[32 * C + lane] = pa;
                if (fb) o1[32 * C + lane] = pb;
                if (lane == 0) {
                    OsjMeta *m0 = (sw ? me1 : me0) + par * 2, *m1 = (sw ? me0 : me1) + par * 2;
                    m0->nrm = a;
                    m0->idx = ix;
                    m0->part = fa;
                    m1->nrm = b;
                    m1->idx = iy;
                    m1->part = fb;
                }
            }
            if (r == N - 2 && lane == 0 && mine) atomicAdd(ctrl + 4 + sweep, mine);
            cl.sync();
            if (active && S > 1) {
                const OsjMeta* m = meta + warp * 4 + par * 2;
                const int i0 = m[0].idx, i1 = m[1].idx;
                sw = i1 < i0;
                ix = min(i0, i1);
                iy = max(i0, i1);
                a = m[sw ? 1 : 0].nrm;
                b = m[sw ? 0 : 1].nrm;
                fa = m[sw ? 1 : 0].part;
                fb = m[sw ? 0 : 1].part;
                const double* in = inbox + ((size_t)warp * 4 + par * 2) * ROW;
                const double *f0 = in + (sw ? ROW : 0), *f1 = in + (sw ? 0 : ROW);
#pragma unroll
                for (int e = 0; e < C; ++e) {
                    x[e] = f0[lane + 32 * e];
                    y[e] = f1[lane + 32 * e];
                }
                pa = f0[32 * C + lane];
                pb = f1[32 * C + lane];
            }
        }
        // N - 1 rounds, an odd number: the next sweep writes parity 0, just read
        done = __ldcg(ctrl + 4 + sweep) == 0;
        cl.sync();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctrl[2] = k >= 2 ? sweep : 0;
        if (!done) atomicOr(status, DEV_NOT_CONVERGED);
    }
    // eigenvalues: the converged rows' squared norms, summed from the rows
    a = norm2(x);
    b = norm2(y);
    auto put = [&](int i, double nn, const double (&v)[C]) {
        if (!active || i >= k) return;
        const double f = nn > 0.0 ? 1.0 / sqrt(nn) : 0.0;
        if (lane == 0) lam_u[i] = nn;
#pragma unroll
        for (int e = 0; e < C; ++e)
            if (lane + 32 * e < n) vt_u[(long)i * n + lane + 32 * e] = f * v[e];
    };
    put(ix, a, x);
    put(iy, b, y);
    for (int i = k + blockIdx.x * wpb + warp; i < n; i += gridDim.x * wpb) {
        if (lane == 0) lam_u[i] = 0.0;
        for (int j = lane; j < n; j += 32) vt_u[(long)i * n + j] = 0.0;
    }
}

__global__ void __launch_bounds__(32 * OSJ_MAX_WARPS, 1)
osj_cluster_kernel(int n, const int* __restrict__ k_dev, const double* W, double* lam_u, double* vt_u, int* ctrl,
                   int* status, int max_sweeps, const int* n_dev, int nsmall) {
    if (n_dev) {  // a captured step: larger sizes take the grid kernel
        n = *n_dev;
        if (n > nsmall) return;  // every CTA, before any barrier
    }
    extern __shared__ double osj_inbox[];
    const double tol = sqrt((double)n) * 2.220446049250313e-16;  // as in osj_kernel
    const int kraw = *k_dev;
    if (kraw < 0) {
        const int wpb = blockDim.x >> 5, lane = threadIdx.x & 31;
        for (int i = blockIdx.x * wpb + (threadIdx.x >> 5); i < n; i += gridDim.x * wpb) {
            if (lane == 0) lam_u[i] = __longlong_as_double(0x7ff8000000000000LL);
            for (int j = lane; j < n; j += 32) vt_u[(long)i * n + j] = 0.0;
        }
        return;
    }
    const int k = min(kraw, n);
#define OSJ_BODY(C) osj_cluster_body<C>(n, k, W, lam_u, vt_u, ctrl, status, max_sweeps, tol, osj_inbox)
    switch ((n + 31) / 32) {
        case 0:
        case 1: OSJ_BODY(1); break;
        case 2: OSJ_BODY(2); break;
        case 3: OSJ_BODY(3); break;
        case 4: OSJ_BODY(4); break;
        case 5: OSJ_BODY(5); break;
        case 6: OSJ_BODY(6); break;
        case 7: OSJ_BODY(7); break;
        default: OSJ_BODY(8); break;
    }
#undef OSJ_BODY
}

// OSJ_CLUSTER_N < n <= OSJ_GRID_N: the same rotations with the rows in L2, over all
// SMs.  A sub-partition issues an FP64 warp instruction in 64 clocks and an SM has
// four, so a CTA is four warps and a pair takes as many of them as there are:
// G = 4 with one pair a CTA, 2 with two, else 1 (a warp's entries of a row:
// n / (32 G)).  With a warp a pair and 32 entries a lane whatever n, a round of
// 451 rows of 713 took 11.8 us.
// There is no grid barrier between rounds.  A round's pairs are round_pair's, in
// which a slot's two rows come from the slots beside it, so a pair waits for its two
// neighbours' count of finished rounds (a store with release, a load with acquire)
// and a slow pair delays only those near it.  Every CTA is resident (cooperative
// launch) and every wait is bounded: a warp whose wait ran out sets DEV_TIMEOUT
// and waits no more, and the grid barrier after the sweep ends the kernel.
// nrm[i]: row i's squared norm, or -1 where part[i] holds its partial sums, to be
// summed over the lanes with the next inner product.  Of a rotation's two new norms
// the shrinking one is summed again only where it halved, an eighth of the FP64
// instructions of a rotating pair less (rank 451 of 713: 34 -> 31 ms).
// Measured (GB300, factorisation included): graded full-rank matrices n = 300 25.1 ->
// 14.0 ms, 449 39.2 -> 31.5, 608 76.8 -> 48.8; rank 451 of 713 47 -> 34; rank 311
// of 311 20 -> 12.
constexpr int OSJ_GRID_N = 1024;
constexpr int OSJ_FLAG = 8;  // ints between two slots' counts: a sector each

template <int E, int G>
__device__ bool osj_grid_body(int n, int k, double* W, double* nrm, double* part, int* flags, int* ctrl, int* status,
                              int max_sweeps, double tol, int& sweeps) {
    __shared__ double s_red[4][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int N = k + (k & 1), S = N / 2;
    const int b = (S + gridDim.x - 1) / gridDim.x;  // pairs of a CTA, at most 4 / G
    const int g = warp / G, w = warp % G, slot = blockIdx.x * b + g;
    const bool active = g < b && slot < S;
    const int ne = (n + 32 * G - 1) / (32 * G);
    int* mine_flag = flags + (long)slot * OSJ_FLAG;
    const int* near = flags + (long)(slot + (lane & 1 ? 1 : -1)) * OSJ_FLAG;  // lanes 0 and 1 watch the neighbours
    const bool watch = active && lane < 2 && (lane & 1 ? slot + 1 < S : slot > 0);
    auto group_sync = [&]() {
        if (G == 1)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(32 * G) : "memory");
    };
    // sums over the pair's warps of up to three values
    auto across = [&](int m, double& v0, double& v1, double& v2) {
        if (G == 1) return;
        if (lane == 0) {
            s_red[warp][0] = v0;
            if (m > 1) {
                s_red[warp][1] = v1;
                s_red[warp][2] = v2;
            }
        }
        group_sync();
        const int w0 = g * G, i = lane & 3;  // a lane a value
        double u = s_red[w0][i] + s_red[w0 + 1][i];
        if (G == 4) u += s_red[w0 + (G == 4 ? 2 : 0)][i] + s_red[w0 + (G == 4 ? 3 : 0)][i];
        v0 = __shfl_sync(0xffffffffu, u, 0);
        if (m > 1) {
            v1 = __shfl_sync(0xffffffffu, u, 1);
            v2 = __shfl_sync(0xffffffffu, u, 2);
        }
    };
    if (active && w == 0 && lane == 0) *mine_flag = 0;
    unsigned epoch = 0;
    if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return false;
    bool late = false, done = k < 2;
    int sweep = 0, round = 0;  // round: rounds since the kernel's start
    for (; sweep < max_sweeps && !done; ++sweep) {
        int mine = 0;
        for (int r = 0; active && r < N - 1; ++r, ++round) {
            if (r > 0 && !late) {
                int it = 0;
                while (!__all_sync(0xffffffffu, !watch || (int)ld_acquire(reinterpret_cast<const unsigned*>(near)) >= round)) {
                    if (++it > SPIN_LIMIT) {
                        late = true;
                        if (lane == 0) atomicOr(status, DEV_TIMEOUT);
                        break;
                    }
                }
                __syncwarp();
            }
            int p, q;
            round_pair(N, r, slot, p, q);
            const bool both = q < k;
            double* wp = W + (long)p * n + 32 * w + lane;
            double* wq = W + (long)q * n + 32 * w + lane;
            double x[E], y[E];
            bool rot = false;
            if (both) {
                const int left = n - 32 * w - lane;  // columns from this lane's first
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (e < ne) {
                        x[e] = 32 * G * e < left ? __ldcg(wp + 32 * G * e) : 0.0;
                        y[e] = 32 * G * e < left ? __ldcg(wq + 32 * G * e) : 0.0;
                    }
                double a = __ldcg(nrm + p), bb = __ldcg(nrm + q);
                double pa = __ldcg(part + (long)p * 128 + 32 * w + lane), pb = __ldcg(part + (long)q * 128 + 32 * w + lane);
                double c0 = 0.0, c1 = 0.0;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (e < ne) {
                        if (e & 1)
                            c1 = fma(x[e], y[e], c1);
                        else
                            c0 = fma(x[e], y[e], c0);
                    }
                double c = c0 + c1;
                bool fa = a < 0.0, fb = bb < 0.0;
                if (r == 0) {  // norms summed afresh at every sweep
                    pa = pb = 0.0;
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (e < ne) {
                            pa = fma(x[e], x[e], pa);
                            pb = fma(y[e], y[e], pb);
                        }
                    fa = fb = true;
                }
                const bool sums = fa || fb;
                if (sums) {
                    osj_sum3(c, pa, pb, lane);
                    across(3, c, pa, pb);
                    a = fa ? pa : a;
                    bb = fb ? pb : bb;
                } else {
                    c = warp_sum(c);
                    across(1, c, pa, pb);
                }
                if (a > 0.0 && bb > 0.0) {
                    const int far = osj_far(c, a, bb, tol);
                    rot = far > 0 || (far == 0 && fabs(c) > tol * sqrt(a * bb));
                }
                if (rot) {
                    double t, cs, sn;
                    osj_angle(a, bb, c, t, cs, sn);
                    // the shrinking row's norm is summed again only where it lost
                    // more than half (the formula cancels no further)
                    const double tc = t * c;
                    const bool p_shrinks = tc > 0.0;
                    const double old = p_shrinks ? a : bb;
                    a -= tc;
                    bb += tc;
                    const bool resum = __double2hiint(p_shrinks ? a : bb) < __double2hiint(old) - (1 << 20);
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (e < ne) {
                            const double xn = cs * x[e] - sn * y[e];
                            y[e] = sn * x[e] + cs * y[e];
                            x[e] = xn;
                            if (32 * G * e < left) {
                                __stcg(wp + 32 * G * e, x[e]);
                                __stcg(wq + 32 * G * e, y[e]);
                            }
                        }
                    if (resum) {
                        double ns = 0.0;
#pragma unroll
                        for (int e = 0; e < E; ++e)
                            if (e < ne) {
                                const double v = p_shrinks ? x[e] : y[e];
                                ns = fma(v, v, ns);
                            }
                        __stcg(part + (long)(p_shrinks ? p : q) * 128 + 32 * w + lane, ns);
                        if (p_shrinks)
                            a = -1.0;
                        else
                            bb = -1.0;
                    }
                    ++mine;
                }
                if ((rot || sums) && w == 0 && lane == 0) {
                    __stcg(nrm + p, a);
                    __stcg(nrm + q, bb);
                }
            } else if (r == 0) {  // the row that sits a round out
                double ns = 0.0;
                for (int j = 32 * w + lane; j < n; j += 32 * G) {
                    const double v = __ldcg(W + (long)p * n + j);
                    ns = fma(v, v, ns);
                }
                __stcg(part + (long)p * 128 + 32 * w + lane, ns);
                if (w == 0 && lane == 0) __stcg(nrm + p, -1.0);
            }
            group_sync();
            if (w == 0 && lane == 0)
                asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(mine_flag), "r"(round + 1) : "memory");
        }
        if (active && w == 0 && lane == 0 && mine) atomicAdd(ctrl + 4 + sweep, mine);
        if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return false;
        done = __ldcg(ctrl + 4 + sweep) == 0;
    }
    sweeps = k >= 2 ? sweep : 0;
    if (!done && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, DEV_NOT_CONVERGED);
    return true;
}

__global__ void __launch_bounds__(128, 1)
osj_grid_kernel(int n, const int* __restrict__ k_dev, double* W, double* nrm, double* lam_u, double* vt_u, int* ctrl,
                int* status, int max_sweeps, const int* n_dev, int nsmall, int nlarge, double* part, int* flags) {
    if (n_dev) {  // a captured step: other sizes take the launches beside it
        n = *n_dev;
        if (n <= nsmall || n > nlarge) return;  // every CTA, before any barrier
    }
    const double tol = sqrt((double)n) * 2.220446049250313e-16;  // as in osj_kernel
    const int lane = threadIdx.x & 31, gw = blockIdx.x * 4 + (threadIdx.x >> 5), nw = gridDim.x * 4;
    const int kraw = *k_dev;
    const int k = min(kraw, n);
    int sweeps = 0;
    if (kraw >= 0) {
        const int b = ((k + 1) / 2 + gridDim.x - 1) / gridDim.x;
        bool ok;
        if (b <= 1)
            ok = osj_grid_body<OSJ_GRID_N / 128, 4>(n, k, W, nrm, part, flags, ctrl, status, max_sweeps, tol, sweeps);
        else if (b == 2)
            ok = osj_grid_body<OSJ_GRID_N / 64, 2>(n, k, W, nrm, part, flags, ctrl, status, max_sweeps, tol, sweeps);
        else
            ok = osj_grid_body<OSJ_GRID_N / 32, 1>(n, k, W, nrm, part, flags, ctrl, status, max_sweeps, tol, sweeps);
        if (!ok) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) ctrl[2] = sweeps;
    }
    // eigenvalues: the converged rows' squared norms, summed from the rows
    for (int i = gw; i < n; i += nw) {
        double a = 0.0;
        if (i < k) {
            for (int j = lane; j < n; j += 32) {
                const double v = __ldcg(W + (long)i * n + j);
                a = fma(v, v, a);
            }
            a = warp_sum(a);
        }
        const double f = a > 0.0 ? 1.0 / sqrt(a) : 0.0;
        if (lane == 0) lam_u[i] = kraw < 0 ? __longlong_as_double(0x7ff8000000000000LL) : a;
        for (int j = lane; j < n; j += 32) vt_u[(long)i * n + j] = i < k ? f * __ldcg(W + (long)i * n + j) : 0.0;
    }
}

// Pivoted Cholesky on one thread-block cluster for n <= PCHOL_SMALL_N: the
// same factorisation as pchol_kernel (pivot = largest remaining diagonal
// entry, ties to the lowest index, stop at the floor, -inf marks pivoted
// columns), with contiguous blocks of cpc columns per CTA whose part of W lies
// in its shared memory (column by column, PCHOL_LD apart).  A column is four
// lanes, one for each of the four interleaved sums of its inner product with
// the pivot column.  A pivot:
//   1. every warp reads the candidates that all column warps have sent to its
//      CTA and takes the same pivot p (integer maxima: a positive double's bits
//      order as its value);
//   2. the CTA copies W[0..k)[p] from the owner's shared memory;
//   3. the column warps form the inner products while a warp without columns
//      takes the square root;
//   4. row k of W, the residual diagonal, and each warp's next candidate, sent
//      to every CTA; one hardware cluster barrier (release / acquire).
// On GB300 a DFMA holds its warp 64 clocks and a barrier costs about 400, so a
// pivot is a chain of k / 4 DFMAs and some 2,000 clocks of the rest; one lane
// per column took k DFMAs in a row.  Candidate slots alternate with the pivot's
// parity, so no CTA overwrites one that another may still read.
// Measured (GB300, one factorisation): n = 61 0.52 -> 0.34 ms, 163 1.44 -> 0.65,
// 256 2.77 -> 1.07, 384 5.4 -> 1.9; above, against pchol_kernel, 449 3.2 -> 2.4 and
// 600 4.5 -> 3.9 (the FMAs of larger sizes want more than a cluster).
constexpr int PCHOL_SMALL_N = 608;
constexpr int PCHOL_SLOTS = 112;  // column warps of a cluster

__host__ __device__ inline int pchol_ld(int n) { return (n + 15) / 16 * 16 + 4; }  // columns 4 banks of 16 apart
__host__ __device__ inline size_t pchol_smem_doubles(int n, int cpc) { return (size_t)cpc * pchol_ld(n) + n; }

__global__ void __launch_bounds__(256)
pchol_cluster_kernel(int n, int cpc, const double* __restrict__ G, long ldg, double* W, int* kB_out,
                     double floor_rel, const int* n_dev, int nsmall) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int CL = (int)cl.num_blocks();
    const int rank = (int)cl.block_rank();
    if (n_dev) {  // a captured step: the size is the device's; larger sizes take pchol_kernel
        n = *n_dev;
        ldg = n;
        if (n > nsmall) return;  // every CTA of the cluster, before any barrier
        if (n <= 0) {
            if (rank == 0 && threadIdx.x == 0) *kB_out = 0;
            return;
        }
        cpc = (n + CL - 1) / CL;
    }
    extern __shared__ double sm[];
    const int ld = pchol_ld(n);
    double* Wl = sm;                         // this CTA's columns: [cpc][ld]
    double* colp = sm + (size_t)cpc * ld;    // W[0..k)[p]
    __shared__ unsigned long long s_key[2][PCHOL_SLOTS];  // candidates of the cluster's column warps, per parity
    __shared__ int s_idx[2][PCHOL_SLOTS];
    __shared__ double s_l;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int cw = (cpc + 7) / 8;  // column warps; the last warp has no columns
    const int c = warp * 8 + (lane >> 2), q = lane & 3;
    const int j = rank * cpc + c;
    const bool own = warp < cw && c < cpc && j < n;
    const int nslots = CL * cw;
    double dj = own ? G[(long)j * ldg + j] : -1.0;
    // this warp's candidate (the largest positive residual, lowest index) to
    // every CTA's slot
    auto post = [&](int par) {
        if (warp >= cw) return;
        unsigned long long key = own && dj > 0.0 ? (unsigned long long)__double_as_longlong(dj) : 0ull;
        const unsigned hi = (unsigned)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
        const unsigned lo = hi == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
        key = (unsigned long long)mh << 32 | ml;
        const int idx = __reduce_min_sync(0xffffffffu, key != 0 && own && hi == mh && lo == ml ? j : n);
        if (lane < CL) {
            *cl.map_shared_rank(&s_key[par][rank * cw + warp], lane) = key;
            *cl.map_shared_rank(&s_idx[par][rank * cw + warp], lane) = idx;
        }
    };
    // the cluster's candidate, from this CTA's slots (after a barrier)
    auto gather = [&](int par, double& d, int& p) {
        unsigned long long key = 0;
        int idx = n;
        for (int i = lane; i < nslots; i += 32) {
            const unsigned long long k2 = s_key[par][i];
            const int i2 = s_idx[par][i];
            if (k2 > key || (k2 == key && i2 < idx)) {
                key = k2;
                idx = i2;
            }
        }
        const unsigned hi = (unsigned)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
        const unsigned lo = hi == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
        p = __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? idx : n);
        d = __longlong_as_double((long long)((unsigned long long)mh << 32 | ml));
    };
    // Inf or NaN on the diagonal (a Gram matrix shows any non-finite entry of
    // its factor there): rank -1 reports it instead of factorising
    const int bad = __syncthreads_or(own && !isfinite(dj));
    cl.sync();  // every CTA of the cluster runs before its shared memory is written
    post(0);
    if (bad && threadIdx.x < CL) *cl.map_shared_rank(&s_key[0][rank * cw], threadIdx.x) = ~0ull;  // marks it
    cl.sync();
    bool anybad = false;
    for (int i = 0; i < nslots; ++i) anybad |= s_key[0][i] == ~0ull;
    if (anybad) {
        if (rank == 0 && threadIdx.x == 0) *kB_out = -1;
        return;
    }
    double dp;
    int p;
    gather(0, dp, p);
    const double floor_abs = floor_rel * dp;
    int par = 0;
    int k = 0;
    for (; k < n; ++k) {
        if (!(dp > floor_abs) || p >= n) break;
        const double g = own && q == 0 ? G[(long)p * ldg + j] : 0.0;
        {
            const double* Wo = cl.map_shared_rank(Wl, p / cpc) + (size_t)(p % cpc) * ld;  // the owner's column
            for (int m = threadIdx.x; m < k; m += blockDim.x) colp[m] = Wo[m];
        }
        __syncthreads();
        double acc = 0.0;
        if (warp < cw) {
            const double* wc = Wl + (size_t)(own ? c : 0) * ld;
            const int k4 = k & ~3;
#pragma unroll 4
            for (int m = q; m < k4; m += 4) acc = fma(colp[m], wc[m], acc);
            if (q == 0)
                for (int m = k4; m < k; ++m) acc = fma(colp[m], wc[m], acc);
            acc += __shfl_down_sync(0xffffffffu, acc, 1, 4);  // lanes 0 and 2: a0 + a1, a2 + a3
            acc += __shfl_down_sync(0xffffffffu, acc, 2, 4);
        } else if (warp == nwarps - 1) {
            const double l = intfp::root(dp);
            if (lane == 0) s_l = l;
        }
        __syncthreads();
        if (own && q == 0) {
            const double l = s_l;
            double w;
            if (j == p) {
                w = l;
                dj = -INFINITY;
            } else if (dj == -INFINITY) {
                w = 0.0;
            } else {
                w = intfp::div(g - acc, l);
                dj = dj - w * w;
            }
            Wl[(size_t)c * ld + k] = w;
            __stcg(W + (long)k * n + j, w);
        }
        if (q != 0) dj = -1.0;  // lane 0 of a column holds its residual
        par ^= 1;
        post(par);
        cl.sync();
        gather(par, dp, p);
    }
    cl.sync();  // no CTA leaves while another may still read its shared memory
    if (rank == 0 && threadIdx.x == 0) *kB_out = k;
}

// One CTA per source row j: rank of lam_j among all (descending, ties by index),
// then copy eigenvector row j and eigenvalue to their sorted positions.
__global__ void __launch_bounds__(256)
jacobi_sort_kernel(int n, const double* __restrict__ d, long ld, const double* __restrict__ vt,
                   double* lam, double* Vt, long ldv, int* sweeps_out, const int* ctrl, const int* n_dev) {
    if (n_dev) {
        n = *n_dev;
        ld = ldv = n;
        if ((int)blockIdx.x >= n) return;
    }
    __shared__ int s_rank[256];
    const int j = blockIdx.x;
    const double lj = d[j];
    int cnt = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double li = d[i];
        if (li > lj || (li == lj && i < j)) ++cnt;
    }
    s_rank[threadIdx.x] = cnt;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s_rank[threadIdx.x] += s_rank[threadIdx.x + o];
        __syncthreads();
    }
    const int rank = s_rank[0];
    if (threadIdx.x == 0) lam[rank] = lj;
    for (int i = threadIdx.x; i < n; i += blockDim.x) Vt[(long)rank * ldv + i] = vt[(long)j * ld + i];
    if (j == 0 && threadIdx.x == 0 && sweeps_out) *sweeps_out = ctrl[2];
}

__global__ void trivial_eig_kernel(const double* G, double* lam, double* Vt, int* sweeps) {
    lam[0] = G[0];
    Vt[0] = 1.0;
    if (sweeps) *sweeps = 0;
}

// ------------------------------------------------------------ pivoted Cholesky
// Left-looking: W[k][j] = (G[p][j] - sum_{m<k} Wc[p][m] Wc[j][m]) / sqrt(d_p) with
// p = argmax of the remaining diagonal d.  W (n x n rows used: k < rank,
// row-major) and its transpose Wc (n x n, Wc[j][m] = W[m][j]) are both written
// so every dot product reads contiguous memory.  d[j] = -inf marks pivoted
// columns; a residual that rounds below zero is only never chosen as a pivot
// (its later entries of W are still formed: treating it as pivoted would drop
// them, up to sqrt(eps_mach) of the pivots' scale each).
// The residual diagonal is double-buffered (2 n entries): step k reads
// d[k & 1] and writes d[(k + 1) & 1], so a CTA that still searches step k's
// pivot never sees another CTA's step-k updates (with one buffer a slow CTA
// could pick a different pivot once the fast ones had marked theirs).
__global__ void __launch_bounds__(JT)
pchol_kernel(int n, const double* __restrict__ G, long ldg, double* W, double* Wc, double* d,
             int* ctrl, int* status, double floor_rel, const int* n_dev, int nsmall) {
    if (n_dev) {  // a captured step: sizes up to nsmall go to pchol_cluster_kernel
        n = *n_dev;
        ldg = n;
        if (n <= nsmall) return;  // every CTA, before any barrier
    }
    unsigned epoch = 0;
    extern __shared__ double sm[];
    double* colp = sm;  // Wc[p][0..k)
    __shared__ double s_val[JT];
    __shared__ int s_idx[JT];
    __shared__ double s_dmax0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    // every CTA reads the initial diagonal (G is an input and is not written)
    double dm = 0.0;
    int bad = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double x = G[(long)j * ldg + j];
        dm = fmax(dm, x);
        bad |= !isfinite(x);
    }
    // Inf or NaN on the diagonal: every CTA reads all of it, so all leave here
    // together (before the first grid barrier) and rank -1 reports it
    if (__syncthreads_or(bad)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) ctrl[3] = -1;
        return;
    }
    s_val[threadIdx.x] = dm;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s_val[threadIdx.x] = fmax(s_val[threadIdx.x], s_val[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) s_dmax0 = s_val[0];
    __syncthreads();
    const double floor_abs = floor_rel * s_dmax0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
        __stcg(d + j, G[(long)j * ldg + j]);
    if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return;
    int k = 0;
    for (; k < n; ++k) {
        const double* dcur = d + (size_t)(k & 1) * n;
        double* dnext = d + (size_t)((k + 1) & 1) * n;
        // argmax of the remaining diagonal (identical in every CTA; ties -> lowest index)
        double best = -1.0;
        int bi = n;
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            const double v = __ldcg(dcur + j);
            if (v > best) {
                best = v;
                bi = j;
            }
        }
        s_val[threadIdx.x] = best;
        s_idx[threadIdx.x] = bi;
        __syncthreads();
        for (int o = blockDim.x / 2; o > 0; o >>= 1) {
            if (threadIdx.x < o) {
                const double v2 = s_val[threadIdx.x + o];
                const int i2 = s_idx[threadIdx.x + o];
                if (v2 > s_val[threadIdx.x] || (v2 == s_val[threadIdx.x] && i2 < s_idx[threadIdx.x])) {
                    s_val[threadIdx.x] = v2;
                    s_idx[threadIdx.x] = i2;
                }
            }
            __syncthreads();
        }
        const double dp = s_val[0];
        const int p = s_idx[0];
        __syncthreads();
        if (!(dp > floor_abs) || p >= n) break;
        const double l = sqrt(dp);
        for (int m = threadIdx.x; m < k; m += blockDim.x) colp[m] = __ldcg(Wc + (long)p * n + m);
        __syncthreads();
        // this CTA's columns j = blockIdx.x + c * gridDim.x, one warp per column
        for (int j = blockIdx.x + warp * gridDim.x; j < n; j += nwarps * gridDim.x) {
            const double dj = __ldcg(dcur + j);
            const bool pivoted = dj == -INFINITY;
            double acc = 0.0;
            if (!pivoted && j != p)
                for (int m = lane; m < k; m += 32) acc += colp[m] * __ldcg(Wc + (long)j * n + m);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) {
                double w;
                if (j == p) {
                    w = l;
                    __stcg(dnext + j, -INFINITY);
                } else if (pivoted) {
                    w = 0.0;
                    __stcg(dnext + j, dj);
                } else {
                    w = (G[(long)p * ldg + j] - acc) / l;
                    __stcg(dnext + j, dj - w * w);
                }
                __stcg(W + (long)k * n + j, w);
                __stcg(Wc + (long)j * n + k, w);
            }
        }
        if (!grid_barrier(ctrl, status, gridDim.x, epoch)) return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl[3] = k;
}

__global__ void pchol_finish_kernel(const int* ctrl, int* kB_out, const int* n_dev, int nsmall) {
    if (n_dev && *n_dev <= nsmall) return;
    *kB_out = ctrl[3];
}

// Self-test of the bounded wait: one CTA enters grid_barrier claiming a grid
// of two, so the second arrival never comes; the wait runs out after its
// iteration limit (~1 s), latches DEV_TIMEOUT and the kernel returns.
__global__ void wait_probe_kernel(int* ctrl, int* status) {
    unsigned epoch = 0;
    if (grid_barrier(ctrl, status, 2u, epoch) && threadIdx.x == 0) atomicOr(status, 0);
}

// The rank of a bond.  One running sum from the small end serves the total, the
// search for the rank (all sums at once) and the discarded tail; it is one chain of
// FP64 additions from shared memory (up to TRUNC_N eigenvalues).  Read from global
// memory by one thread, three times over, it took 20 us at 126 to 163 eigenvalues
// (GB300), now 7.
constexpr int TRUNC_N = 2048;
__global__ void __launch_bounds__(256)
truncation_kernel(const double* lamK, int kB, double eps, int dm1, int forced,
                  int max_rank, double* delta2_dev, int* dec_i, double* dec_d,
                  const int* kB_dev, int sv) {
    if (kB_dev) kB = *kB_dev > 0 ? *kB_dev : 0;
    const double eps_mach = 2.220446049250313e-16;
    __shared__ double S[TRUNC_N];  // sums of lamK[j], j from kB - 1 down to the index
    __shared__ double s_delta2;
    __shared__ int s_avail, s_above;
    const bool fit = kB <= TRUNC_N;
    double total = 0.0;
    if (threadIdx.x == 0) {
        s_avail = 0;
        s_above = -1;
    }
    for (int j = threadIdx.x; fit && j < kB; j += blockDim.x) S[j] = lamK[j];
    __syncthreads();
    if (threadIdx.x == 0) {
        // totals and tails are summed from the small end; eigenvalues are not clamped
        // at zero, so the symmetric rounding noise of the Gram eigenvalues cancels
        for (int j = kB - 1; j >= 0; --j) {
            total += fit ? S[j] : lamK[j];
            if (fit) S[j] = total;
        }
        // an Inf or NaN anywhere in the tensor reaches the eigenvalues (or their
        // sum); the host reports it instead of rounding to the zero tensor
        dec_i[2] = isfinite(total) ? 0 : 1;
        total = fmax(total, 0.0);
        double delta2 = *delta2_dev;
        if (delta2 < 0.0) {
            delta2 = eps * eps * total / (double)(dm1 > 0 ? dm1 : 1);
            *delta2_dev = delta2;
        }
        s_delta2 = delta2;
    }
    __syncthreads();
    const double delta2 = s_delta2;
    // floor: Gram eigenvalues are resolved to kB eps_mach of the largest;
    // squared singular values from an SVD (sv) to the square of that
    const double lmax = kB > 0 ? lamK[0] : 0.0;
    const double fl = sv ? ((double)kB * eps_mach) * ((double)kB * eps_mach) : (double)kB * eps_mach;
    // above: the first sum from the small end that exceeds delta^2
    int avail = 0, above = -1;
    for (int j = threadIdx.x; j < kB; j += blockDim.x) {
        if (lmax > 0.0 && lamK[j] > fl * lmax) ++avail;
        if (fit && S[j] > delta2) above = j;
    }
    if (avail) atomicAdd(&s_avail, avail);
    if (above >= 0) atomicMax(&s_above, above);
    if (!fit && threadIdx.x == 0) {
        double t = 0.0;
        for (int j = kB - 1; j >= 0; --j) {
            t += lamK[j];
            if (t > delta2) {
                atomicMax(&s_above, j);
                break;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const int navail = s_avail;
    int r, capped = 0;
    if (navail == 0) {
        r = 0;
    } else if (forced > 0) {
        r = min(forced, navail);
    } else {
        // smallest r >= 1 with sum_{j >= r} sigma_j^2 <= delta^2
        r = max(1, s_above + 1);
        if (max_rank > 0 && r > max_rank) {
            r = max_rank;
            capped = 1;
        }
        r = min(r, navail);
    }
    double tail = 0.0;
    if (fit)
        tail = r < kB ? S[r] : 0.0;
    else
        for (int j = kB - 1; j >= r; --j) tail += lamK[j];
    dec_i[0] = r;
    dec_i[1] = capped;
    dec_d[0] = delta2;
    dec_d[1] = fmax(tail, 0.0);
    dec_d[2] = total;
}

__global__ void count_floor_kernel(const double* lam, int n, int* out) {
    const double eps_mach = 2.220446049250313e-16;
    int cnt = 0;
    const double lmax = n > 0 ? lam[0] : 0.0;
    if (lmax > 0.0)
        for (int j = 0; j < n; ++j)
            if (lam[j] > (double)n * eps_mach * lmax) ++cnt;
    *out = cnt;
}

tt_status coop_blocks(const void* fn, size_t smem, int want, int* out) {
    int dev = 0, sms = 0, per_sm = 0;
    TT_CUDA_TRY(cudaGetDevice(&dev));
    TT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    TT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, JT, smem));
    if (per_sm < 1) {
        set_error("persistent kernel cannot be resident with its shared memory");
        return TT_ERR_CUDA;
    }
    *out = std::max(1, std::min(want, std::min(sms, per_sm * sms)));
    return TT_OK;
}

tt_status ensure_ctrl(EigWork& w, cudaStream_t s) {
    if (!w.d_ctrl) {
        TT_TRY(w.ctrl_buf.ensure((CTRL_INTS * sizeof(int) + 7) / 8, s));
        w.d_ctrl = reinterpret_cast<int*>(w.ctrl_buf.p);
        w.ctrl_cap = CTRL_INTS;
    }
    TT_CUDA_TRY(cudaMemsetAsync(w.d_ctrl, 0, CTRL_INTS * sizeof(int), s));
    return TT_OK;
}

}  // namespace

void EigWork::release() {
    cs.release();
    g0.release();
    g1.release();
    lam_unsorted.release();
    vt_unsorted.release();
    abc.release();
    psd.release();
    ctrl_buf.release();
    d_ctrl = nullptr;
    ctrl_cap = 0;
}

tt_status syev(cudaStream_t s, int n, const double* G, long ldg, double* lam, double* Vt, long ldv,
               EigWork& w, int* status_dev, int* sweeps_dev, int max_sweeps) {
    if (n < 0) {
        set_error("syev: negative size");
        return TT_ERR_ARG;
    }
    if (max_sweeps < 1 || max_sweeps > MAX_SWEEPS) {
        set_error("syev: the sweep limit must be in 1 .. " + std::to_string(MAX_SWEEPS));
        return TT_ERR_ARG;
    }
    if (n == 0) return TT_OK;
    if (n == 1) {
        note_launch();
        trivial_eig_kernel<<<1, 1, 0, s>>>(G, lam, Vt, sweeps_dev);
        TT_CUDA_TRY(cudaGetLastError());
        return TT_OK;
    }
    // relative skip test as in high-relative-accuracy Jacobi; the absolute one
    // (1e-20 of the largest diagonal entry) only skips rotations inside the
    // block of eigenvalues below the Gram floor n eps_mach lambda_max that the
    // rounding discards afterwards: on the rounding's K matrices it ends the
    // iteration 1-3 sweeps earlier than 1e-24 with the same eigenpairs above
    // the floor.  (One CTA would save the grid barrier per round but not the
    // round's ~n^2 FP64 FMAs, which one SM's share of GB300's FP64 rate cannot
    // absorb: measured 1.1 ms mean per eigensolve at n <= 96.)
    double tol_rel = 1e-15, tol_abs_rel = 1e-20;
    const int N = n + (n & 1);
    const int npairs = N / 2;
    const long ld = n;
    TT_TRY(w.g0.ensure((size_t)n * n, s));
    TT_TRY(w.g1.ensure((size_t)n * n, s));
    TT_TRY(w.vt_unsorted.ensure((size_t)n * n, s));
    TT_TRY(w.lam_unsorted.ensure((size_t)n, s));
    TT_TRY(w.abc.ensure((size_t)6 * npairs, s));
    TT_TRY(w.cs.ensure((size_t)2 * npairs, s));
    TT_TRY(ensure_ctrl(w, s));
    // one row pair per CTA where the GPU holds that many CTAs: a round's FP64
    // work per CTA (about 18 n flops per owned pair) is what bounds the round
    // on GB300's FP64 pipe, so the pairs are spread over as many SMs as exist.
    // Shared memory: all angles, the owned rows, the list of active pairs.
    auto smem_for = [&](int ppc) {
        return (size_t)(npairs * 2 + 2 * (size_t)ppc * n) * sizeof(double) + (size_t)npairs * sizeof(int);
    };
    int want = npairs;
    // the row buffers for MAX_PAIRS_PER_CTA pairs where they fit; above that
    // (n > ~1480) for the pairs each SM must own
    size_t smem = smem_for(MAX_PAIRS_PER_CTA);
    if (smem > 200 * 1024) {
        int dev = 0, sms = 1;
        TT_CUDA_TRY(cudaGetDevice(&dev));
        TT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        smem = smem_for(std::min(MAX_PAIRS_PER_CTA, (npairs + sms - 1) / sms));
    }
    if (smem > 200 * 1024) {
        set_error("syev: matrix too large for the shared-memory row buffers");
        return TT_ERR_TOO_LARGE;
    }
    TT_TRY(ensure_max_dynamic_smem((const void*)jacobi_kernel));
    int blocks = 1;
    TT_TRY(coop_blocks((const void*)jacobi_kernel, smem, want, &blocks));
    const int ppc = (npairs + blocks - 1) / blocks;
    if (ppc > MAX_PAIRS_PER_CTA || smem_for(ppc) > smem) {
        set_error("syev: too few resident CTAs for this matrix size");
        return TT_ERR_TOO_LARGE;
    }
    {
        const long total = (long)n * n;
        const int ib = (int)std::min<long>((total + 255) / 256, 152L * 16);
        note_launch();
        jacobi_init_kernel<<<ib, 256, 0, s>>>(n, N, G, ldg, w.g0.p, w.vt_unsorted.p, ld, w.abc.p, nullptr);
        TT_CUDA_TRY(cudaGetLastError());
    }
    double* g0 = w.g0.p;
    double* g1 = w.g1.p;
    double* vt = w.vt_unsorted.p;
    double* abc0 = w.abc.p;
    double* abc1 = w.abc.p + 3 * npairs;
    double* lamu = w.lam_unsorted.p;
    double* csg = w.cs.p;
    int* ctrl = w.d_ctrl;
    int nn = n, NN = N;
    long ldl = ld;
    int msw = max_sweeps;
    const int* nnull = nullptr;
    void* args[] = {&nn, &NN, &g0, &g1, &ldl, &vt, &abc0, &abc1, &csg, &lamu, &ctrl, &status_dev, &tol_rel,
                    &tol_abs_rel, &msw, &nnull};
    note_launch();
    TT_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)jacobi_kernel, dim3(blocks), dim3(JT), args,
                                            smem, s));
    note_launch();
    jacobi_sort_kernel<<<n, 256, 0, s>>>(n, w.lam_unsorted.p, ld, w.vt_unsorted.p, lam, Vt, ldv,
                                         sweeps_dev, w.d_ctrl, nullptr);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

// Largest cluster (16, else 8) the GPU schedules for a kernel of `threads`
// threads and no dynamic shared memory, found once per kernel.
int cluster_size_for(const void* fn, int threads) {
    static std::mutex mu;
    static std::vector<std::pair<const void*, int>> known;
    std::lock_guard<std::mutex> lock(mu);
    for (auto& kv : known)
        if (kv.first == fn) return kv.second;
    int cl = 8;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = 160 * 1024;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, fn, &cfg) == cudaSuccess && nc > 0) cl = 16;
    }
    (void)cudaGetLastError();
    known.emplace_back(fn, cl);
    return cl;
}

// Largest n the cluster factorisation takes: at most PCHOL_SMALL_N, its columns
// of W in a CTA's shared memory, at most 7 column warps a CTA, a candidate slot
// for each of the cluster's.
int pchol_small_limit() {
    const int cl = cluster_size_for((const void*)pchol_cluster_kernel, 256);
    int n = PCHOL_SMALL_N;
    while (n > 0 && (pchol_smem_doubles(n, (n + cl - 1) / cl) * sizeof(double) > 200 * 1024 ||
                     cl * (((n + cl - 1) / cl + 7) / 8) > PCHOL_SLOTS || ((n + cl - 1) / cl + 7) / 8 > 7))
        --n;
    return n;
}

tt_status launch_pchol_cluster(cudaStream_t s, int n, const double* G, long ldg, double* W, int* kB_dev,
                               const int* n_dev, int nsmall) {
    const int cl = cluster_size_for((const void*)pchol_cluster_kernel, 256);
    const int cpc = (n + cl - 1) / cl;
    const int threads = 32 * std::max(4, (cpc + 7) / 8 + 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = pchol_smem_doubles(n, cpc) * sizeof(double);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // stop at the rounding-noise level of G's entries (eps_mach max diag)
    const double fr = 2.220446049250313e-16;
    note_launch();
    TT_CUDA_TRY(cudaLaunchKernelEx(&cfg, pchol_cluster_kernel, n, cpc, G, ldg, W, kB_dev, fr, n_dev, nsmall));
    return TT_OK;
}

tt_status osj_launch(cudaStream_t s, int ncap, const int* k_dev, EigWork& w, int* status_dev, int max_sweeps,
                     const int* n_dev, double* nrm) {
    TT_TRY(ensure_ctrl(w, s));  // zero barrier and sweep counters (pchol used them)
    int nn = ncap;
    double* Wp = w.g0.p;
    double* lamu = w.lam_unsorted.p;
    double* vtu = w.vt_unsorted.p;
    int* ctrl = w.d_ctrl;
    int msw = max_sweeps;
    int nsmall = OSJ_CLUSTER_N;
    if (ncap <= nsmall || n_dev) {
        // one cluster, a warp per pair.
        // A captured step launches it for sizes up to nsmall and the grid
        // kernel after it for larger ones (each returns at once outside its
        // range), so a replay takes the host path's kernel.
        const int ncl = std::min(ncap, nsmall);
        const int cl = cluster_size_for((const void*)osj_cluster_kernel, 32 * OSJ_MAX_WARPS);
        const int wpb = std::max(1, ((ncl + 1) / 2 + cl - 1) / cl);
        const int C = (ncl + 31) / 32;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cl);
        cfg.blockDim = dim3(32 * wpb);
        cfg.dynamicSmemBytes = (size_t)wpb * 4 * (32 * (C + 1) * sizeof(double) + sizeof(OsjMeta));
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cl;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        note_launch();
        TT_CUDA_TRY(cudaLaunchKernelEx(&cfg, osj_cluster_kernel, nn, k_dev, (const double*)Wp, lamu, vtu, ctrl,
                                       status_dev, msw, n_dev, nsmall));
        if (ncap <= nsmall) return TT_OK;
    }
    int dev = 0, sms = 0;
    TT_CUDA_TRY(cudaGetDevice(&dev));
    TT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    auto resident = [&](const void* fn, int threads, int& blocks) -> tt_status {
        int per_sm = 0;
        TT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, 0));
        if (per_sm < 1) {
            set_error("one-sided Jacobi kernel cannot be resident");
            return TT_ERR_CUDA;
        }
        blocks = per_sm * sms;
        return TT_OK;
    };
    int blocks = 1;
    int nlarge = std::min(OSJ_GRID_N, 8 * sms);  // at most four pairs a CTA
    if (ncap <= nlarge || n_dev) {
        // a CTA per SM whatever n: the pairs' split over warps follows from it and
        // from the rank alone, so a replay's sums are the host path's.  Scratch:
        // pchol's, free by now
        const void* fn = (const void*)osj_grid_kernel;
        TT_TRY(resident(fn, 128, blocks));
        double* part = w.g1.p;                           // 128 a row
        int* flags = reinterpret_cast<int*>(w.psd.p);  // OSJ_FLAG ints a pair of rows
        void* args[] = {&nn, &k_dev, &Wp, &nrm, &lamu, &vtu, &ctrl, &status_dev, &msw, &n_dev, &nsmall, &nlarge, &part, &flags};
        note_launch();
        TT_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(sms), dim3(128), args, 0, s));
        if (ncap <= nlarge) return TT_OK;
        nsmall = nlarge;
    }
    // one CTA per SM with one warp per pair it owns, so every SM carries the
    // same number of pairs in a round (the round ends at the slowest SM)
    const void* fn = (const void*)osj_kernel;
    const int npairs = (ncap + 1) / 2;
    const int wpb = std::max(1, std::min(OSJ_MAX_WARPS, (npairs + sms - 1) / sms));
    TT_TRY(resident(fn, 32 * wpb, blocks));
    blocks = std::max(1, std::min((npairs + wpb - 1) / wpb, blocks));
    void* args[] = {&nn, &k_dev, &Wp, &nrm, &lamu, &vtu, &ctrl, &status_dev, &msw, &n_dev, &nsmall};
    note_launch();
    TT_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(32 * wpb), args, 0, s));
    return TT_OK;
}

tt_status wait_probe(cudaStream_t s, EigWork& w, int* status_dev) {
    TT_TRY(ensure_ctrl(w, s));
    note_launch();
    wait_probe_kernel<<<1, 32, 0, s>>>(w.d_ctrl, status_dev);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

tt_status pchol(cudaStream_t s, int n, const double* G, long ldg, double* W, double* Wc,
                double* dwork, EigWork& w, int* status_dev, int* kB_dev) {
    if (n <= 0) return TT_OK;
    TT_TRY(ensure_ctrl(w, s));
    const size_t smem = (size_t)n * sizeof(double);
    if (smem > 200 * 1024) {
        set_error("pchol: matrix too large");
        return TT_ERR_TOO_LARGE;
    }
    TT_TRY(ensure_max_dynamic_smem((const void*)pchol_kernel));
    const int nsmall = pchol_small_limit();
    if (n <= nsmall) return launch_pchol_cluster(s, n, G, ldg, W, kB_dev, nullptr, nsmall);
    int blocks = 1;
    // about eight columns per CTA (one warp each)
    TT_TRY(coop_blocks((const void*)pchol_kernel, smem, std::max(1, (n + 7) / 8), &blocks));
    int nn = n;
    long ldgl = ldg;
    const double* Gp = G;
    int* ctrl = w.d_ctrl;
    // stop at the rounding-noise level of G's entries (eps_mach max diag): a
    // higher floor (n eps_mach, LAPACK's default for pivoted Cholesky) drops
    // parts of G_B that still carry tensor components at the 1e-9 level
    double fr = 2.220446049250313e-16;
    const int* nnull = nullptr;
    int nsm = nsmall;
    void* args[] = {&nn, &Gp, &ldgl, &W, &Wc, &dwork, &ctrl, &status_dev, &fr, &nnull, &nsm};
    note_launch();
    TT_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)pchol_kernel, dim3(blocks), dim3(JT), args,
                                            smem, s));
    note_launch();
    pchol_finish_kernel<<<1, 1, 0, s>>>(w.d_ctrl, kB_dev, nullptr, nsmall);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

tt_status eig_reserve(EigWork& w, cudaStream_t s) { return ensure_ctrl(w, s); }

tt_status eig_prepare() {
    TT_TRY(ensure_max_dynamic_smem((const void*)pchol_kernel));
    TT_TRY(ensure_max_dynamic_smem((const void*)jacobi_kernel));
    // cluster attributes set before any capture
    cluster_size_for((const void*)pchol_cluster_kernel, 256);
    cluster_size_for((const void*)osj_cluster_kernel, 32 * OSJ_MAX_WARPS);
    return TT_OK;
}

tt_status pchol_dyn(cudaStream_t s, const int* n_dev, int ncap, const double* G, double* W, double* Wc,
                    double* dwork, EigWork& w, int* status_dev, int* kB_dev) {
    if (ncap <= 0) return TT_OK;
    TT_TRY(ensure_ctrl(w, s));
    const int nsmall = pchol_small_limit();
    TT_TRY(launch_pchol_cluster(s, std::min(ncap, nsmall), G, ncap, W, kB_dev, n_dev, nsmall));
    if (ncap > nsmall) {
        const size_t smem = (size_t)ncap * sizeof(double);
        if (smem > 200 * 1024) {
            set_error("pchol: matrix too large");
            return TT_ERR_TOO_LARGE;
        }
        TT_TRY(ensure_max_dynamic_smem((const void*)pchol_kernel));
        int blocks = 1;
        TT_TRY(coop_blocks((const void*)pchol_kernel, smem, std::max(1, (ncap + 7) / 8), &blocks));
        int nn = ncap;
        long ldgl = ncap;
        const double* Gp = G;
        int* ctrl = w.d_ctrl;
        double fr = 2.220446049250313e-16;
        int nsm = nsmall;
        void* args[] = {&nn, &Gp, &ldgl, &W, &Wc, &dwork, &ctrl, &status_dev, &fr, &n_dev, &nsm};
        note_launch();
        TT_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)pchol_kernel, dim3(blocks), dim3(JT), args, smem, s));
        note_launch();
        pchol_finish_kernel<<<1, 1, 0, s>>>(w.d_ctrl, kB_dev, n_dev, nsmall);
        TT_CUDA_TRY(cudaGetLastError());
    }
    return TT_OK;
}

tt_status syev_dyn(cudaStream_t s, const int* n_dev, int ncap, const double* G, double* lam, double* Vt,
                   EigWork& w, int* status_dev, int* sweeps_dev, int max_sweeps) {
    if (ncap <= 0) return TT_OK;
    double tol_rel = 1e-15, tol_abs_rel = 1e-20;
    const int Ncap = ncap + (ncap & 1);
    const int npcap = Ncap / 2;
    TT_TRY(w.g0.ensure((size_t)ncap * ncap, s));
    TT_TRY(w.g1.ensure((size_t)ncap * ncap, s));
    TT_TRY(w.vt_unsorted.ensure((size_t)ncap * ncap, s));
    TT_TRY(w.lam_unsorted.ensure((size_t)ncap, s));
    TT_TRY(w.abc.ensure((size_t)6 * npcap, s));
    TT_TRY(w.cs.ensure((size_t)2 * npcap, s));
    TT_TRY(ensure_ctrl(w, s));
    // grid and shared memory for the largest n; a smaller n leaves CTAs with
    // fewer (or no) pairs, and every pair's arithmetic is the same as in syev
    auto smem_for = [&](int ppc) {
        return (size_t)(npcap * 2 + 2 * (size_t)ppc * ncap) * sizeof(double) + (size_t)npcap * sizeof(int);
    };
    size_t smem = smem_for(MAX_PAIRS_PER_CTA);
    if (smem > 200 * 1024) smem = smem_for(1);
    if (smem > 200 * 1024) {
        set_error("syev: matrix too large for the shared-memory row buffers");
        return TT_ERR_TOO_LARGE;
    }
    TT_TRY(ensure_max_dynamic_smem((const void*)jacobi_kernel));
    int blocks = 1;
    TT_TRY(coop_blocks((const void*)jacobi_kernel, smem, npcap, &blocks));
    const int ppc = (npcap + blocks - 1) / blocks;
    if (ppc > MAX_PAIRS_PER_CTA || smem_for(ppc) > smem) {
        set_error("syev: too few resident CTAs for this matrix size");
        return TT_ERR_TOO_LARGE;
    }
    {
        const long total = (long)ncap * ncap;
        const int ib = (int)std::min<long>((total + 255) / 256, 152L * 16);
        note_launch();
        jacobi_init_kernel<<<ib, 256, 0, s>>>(ncap, Ncap, G, ncap, w.g0.p, w.vt_unsorted.p, ncap, w.abc.p, n_dev);
        TT_CUDA_TRY(cudaGetLastError());
    }
    double* g0 = w.g0.p;
    double* g1 = w.g1.p;
    double* vt = w.vt_unsorted.p;
    double* abc0 = w.abc.p;
    double* abc1 = w.abc.p + 3 * npcap;
    double* csg = w.cs.p;
    double* lamu = w.lam_unsorted.p;
    int* ctrl = w.d_ctrl;
    int nn = ncap, NN = Ncap;
    long ldl = ncap;
    int msw = max_sweeps;
    void* args[] = {&nn, &NN, &g0, &g1, &ldl, &vt, &abc0, &abc1, &csg, &lamu, &ctrl, &status_dev, &tol_rel,
                    &tol_abs_rel, &msw, &n_dev};
    note_launch();
    TT_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)jacobi_kernel, dim3(blocks), dim3(JT), args, smem, s));
    note_launch();
    jacobi_sort_kernel<<<ncap, 256, 0, s>>>(ncap, w.lam_unsorted.p, ncap, w.vt_unsorted.p, lam, Vt, ncap,
                                            sweeps_dev, w.d_ctrl, n_dev);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

void truncation_decision_dyn(cudaStream_t s, const double* lamK, const int* kB_dev, double eps, int dm1,
                             int forced, int max_rank, double* delta2_dev, int* dec_i, double* dec_d) {
    note_launch();
    truncation_kernel<<<1, 256, 0, s>>>(lamK, 0, eps, dm1, forced, max_rank, delta2_dev, dec_i, dec_d, kB_dev, 0);
}

void truncation_decision(cudaStream_t s, const double* lamK, int kB, double eps, int dm1,
                         int forced, int max_rank, double* delta2_dev, int* dec_i,
                         double* dec_d, bool singular_values) {
    note_launch();
    truncation_kernel<<<1, 256, 0, s>>>(lamK, kB, eps, dm1, forced, max_rank, delta2_dev, dec_i,
                                      dec_d, nullptr, singular_values ? 1 : 0);
}

tt_status syev_psd(cudaStream_t s, int n, const double* K, long ldk, double* lam, double* Vt, long ldv,
                   EigWork& w, int* status_dev, int* sweeps_dev, int max_sweeps) {
    if (n < 0) {
        set_error("syev_psd: negative size");
        return TT_ERR_ARG;
    }
    if (max_sweeps < 1 || max_sweeps > MAX_SWEEPS) {
        set_error("syev_psd: the sweep limit must be in 1 .. " + std::to_string(MAX_SWEEPS));
        return TT_ERR_ARG;
    }
    if (n == 0) return TT_OK;
    if (n == 1) {
        note_launch();
        trivial_eig_kernel<<<1, 1, 0, s>>>(K, lam, Vt, sweeps_dev);
        TT_CUDA_TRY(cudaGetLastError());
        return TT_OK;
    }
    TT_TRY(w.g0.ensure((size_t)n * n, s));
    TT_TRY(w.g1.ensure((size_t)n * n, s));
    TT_TRY(w.vt_unsorted.ensure((size_t)n * n, s));
    TT_TRY(w.lam_unsorted.ensure((size_t)n, s));
    TT_TRY(w.psd.ensure((size_t)3 * n + 2, s));
    int* k_dev = reinterpret_cast<int*>(w.psd.p + 3 * n);
    // K = W^T W (pivoted, rows of W in pivot order), then its rows orthogonalised
    TT_TRY(pchol(s, n, K, ldk, w.g0.p, w.g1.p, w.psd.p, w, status_dev, k_dev));
    TT_TRY(osj_launch(s, n, k_dev, w, status_dev, max_sweeps, nullptr, w.psd.p + 2 * n));
    note_launch();
    jacobi_sort_kernel<<<n, 256, 0, s>>>(n, w.lam_unsorted.p, n, w.vt_unsorted.p, lam, Vt, ldv, sweeps_dev,
                                         w.d_ctrl, nullptr);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

tt_status syev_psd_dyn(cudaStream_t s, const int* n_dev, int ncap, const double* K, double* lam, double* Vt,
                       EigWork& w, int* status_dev, int* sweeps_dev, int max_sweeps) {
    if (ncap <= 0) return TT_OK;
    TT_TRY(w.g0.ensure((size_t)ncap * ncap, s));
    TT_TRY(w.g1.ensure((size_t)ncap * ncap, s));
    TT_TRY(w.vt_unsorted.ensure((size_t)ncap * ncap, s));
    TT_TRY(w.lam_unsorted.ensure((size_t)ncap, s));
    TT_TRY(w.psd.ensure((size_t)3 * ncap + 2, s));
    int* k_dev = reinterpret_cast<int*>(w.psd.p + 3 * ncap);
    TT_TRY(pchol_dyn(s, n_dev, ncap, K, w.g0.p, w.g1.p, w.psd.p, w, status_dev, k_dev));
    TT_TRY(osj_launch(s, ncap, k_dev, w, status_dev, max_sweeps, n_dev, w.psd.p + 2 * ncap));
    note_launch();
    jacobi_sort_kernel<<<ncap, 256, 0, s>>>(ncap, w.lam_unsorted.p, ncap, w.vt_unsorted.p, lam, Vt, ncap,
                                            sweeps_dev, w.d_ctrl, n_dev);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

void count_above_floor(cudaStream_t s, const double* lam, int n, int* out_dev) {
    note_launch();
    count_floor_kernel<<<1, 1, 0, s>>>(lam, n, out_dev);
}

}  // namespace ttsn
