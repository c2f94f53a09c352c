// Transport, source and quadrature kernels of the TT-S_N step (arXiv
// 2503.18056, Sec. 3-4) on the paper's three-core layout (Eq. tensor_decomp):
// I_ilp = X_i Theta_l Phi_p, all spatial axes grouped in X (N_c x r1).
//
// Transport (Sec. 4.3): the upwind update of Eq. lhs / Eq. upwind is the TT sum
//   I* = I - sum_a nu_a [ (D^-_a X) (x) (thfac Theta) (x) (phfac Phi)
//                       + (D^+_a X) (x) (thfac' Theta) (x) (phfac' Phi) ],
// nu_a = c dt / dx_a, D^-_a X_i = X_i - X_{i-1}, D^+_a X_i = X_{i+1} - X_i with
// ghost rows per Sec. 4.5 (zero rows for vacuum, wrapped rows for periodic)
// and rank-one masked direction cosines (sin(theta), max/min(cos(phi), 0)) for
// x, (sin(theta), max/min(sin(phi), 0)) for y, (max/min(cos(theta), 0), 1) for
// z.  Terms are summed by TT addition (Sec. 4.1) in the order
// [I, x+, x-, y+, y-, z+, z-]: the spatial core is the concatenation of the
// term cores, the angular cores are block-diagonal / stacked.
//
// Source (Sec. 3.2, 4.4): per cell k_a = c dt sigma_a, k_s = c dt sigma_s,
// E* = X*_i . thbar / c (Eq. tt_energy_density), T-dagger from
// gamma a_r T^4 + T = T^m + gamma E*, gamma = k_a / ((1 + k_a) C_v), then
// I^{m+1} = s I* + e (x) 1 (x) 1 with s = 1/(1 + k_a + k_s) and
// e = s (k_s J^{m+1} + k_a c a_r T-dagger^4 / 4 pi),
// J^{m+1} = (c E*/4 pi + k_a c a_r T-dagger^4 / 4 pi)/(1 + k_a): a row scaling
// of the spatial core plus one appended column (angular cores get a unit
// block), fused into the same pass as transport so the grown spatial core is
// written once.
#include <algorithm>

#include "internal.h"

namespace ttsn {

namespace {

constexpr double FOUR_PI = 12.566370614359172953850573533118;


// Thg: (R1, nt, R2), R1 = nterms r1 + ns (+1 if src), R2 = nterms r2 + ns (+1 if
// src): the term blocks, then one block per external source (its theta
// profile), then the unit block of the emission term.
__global__ void grown_theta_kernel(int nterms, int src, int r1, int r2, int nt, const double* Th,
                                   const double* tfac, int ns,
                                   const double* s_th, double* Thg, int R1, int R2, const int* dd) {
    if (dd) {  // a captured step: ranks from the device's size block
        r1 = dd[DYN_R1];
        r2 = dd[DYN_R2];
        R1 = dd[DYN_G1];
        R2 = dd[DYN_G2];
    }
    const long total = (long)R1 * nt * R2;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int b = (int)(t % R2);
        const long t2 = t / R2;
        const int l = (int)(t2 % nt);
        const int a = (int)(t2 / nt);
        double v = 0.0;
        const int ja = a / r1, jb = b / r2;
        const int ka = a - nterms * r1, kb = b - nterms * r2;
        if (ja == jb && ja < nterms) {
            v = tfac[(long)ja * nt + l] *
                Th[((long)(a - ja * r1) * nt + l) * r2 + (b - jb * r2)];
        } else if (ka >= 0 && ka == kb && ka < ns) {
            v = s_th[(long)ka * nt + l];
        } else if (src && a == R1 - 1 && b == R2 - 1) {
            v = 1.0;
        }
        Thg[t] = v;
    }
}

// Phg: (R2, np)
__global__ void grown_phi_kernel(int nterms, int src, int r2, int np, const double* Ph,
                                 const double* pfac, int ns,
                                 const double* s_ph, double* Phg, int R2, const int* dd) {
    if (dd) {
        r2 = dd[DYN_R2];
        R2 = dd[DYN_G2];
    }
    const long total = (long)R2 * np;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int p = (int)(t % np);
        const int b = (int)(t / np);
        double v = 0.0;
        const int jb = b / r2;
        const int kb = b - nterms * r2;
        if (jb < nterms) {
            v = pfac[(long)jb * np + p] * Ph[(long)(b - jb * r2) * np + p];
        } else if (kb >= 0 && kb < ns) {
            v = s_ph[(long)kb * np + p];
        } else if (src && b == R2 - 1) {
            v = 1.0;
        }
        Phg[t] = v;
    }
}

// phibar[j][b] = sum_p v phfac_j[p] Ph[b][p]
__global__ void phibar_kernel(int nterms, int r2, int np, const double* Ph, const double* pfac, double v, double* phibar,
                              const int* dd) {
    if (dd) r2 = dd[DYN_R2];
    const int total = nterms * r2;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int j = t / r2, b = t % r2;
        double acc = 0.0;
        for (int p = 0; p < np; ++p) acc += pfac[(long)j * np + p] * Ph[(long)b * np + p];
        phibar[t] = v * acc;
    }
}

// thbar[j r1 + a] = sum_l w thfac_j[l] sum_b Th[a][l][b] phibar[j][b]: one warp
// per output, lanes striding over the contiguous (l, b) block of row a.
__global__ void thbar_kernel(int nterms, int r1, int r2, int nt, const double* Th,
                             const double* tfac, double w, const double* phibar,
                             double* thbar, const int* dd) {
    if (dd) {
        r1 = dd[DYN_R1];
        r2 = dd[DYN_R2];
    }
    const int lane = threadIdx.x & 31;
    const int total = nterms * r1;
    const int warps = gridDim.x * (blockDim.x >> 5);
    const int len = nt * r2;
    for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < total; t += warps) {
        const int j = t / r1, a = t % r1;
        const double* row = Th + (long)a * len;
        double acc = 0.0;
        for (int idx = lane; idx < len; idx += 32) {
            const int l = idx / r2, b = idx - l * r2;
            acc += tfac[(long)j * nt + l] * row[idx] * phibar[j * r2 + b];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) thbar[t] = w * acc;
    }
}

// Neighbour rows of cell i along each axis (C order, axis 0 slowest):
// nb[a][0] = lower, nb[a][1] = upper; -1 marks a zero ghost (vacuum edge),
// periodic edges wrap, outflow edges point at the cell itself (Sec. 4.5).
// BC_HALO (axis 0 of a spatial shard, whose layers are the last stride
// rows): the ghost layers are halo rows held after the shard's own nc rows,
// the lower ghost layer at rows nc .. nc + stride - 1 and the upper one after
// it, so a ghost is never a negative (vacuum) index.
__device__ __forceinline__ void cell_neighbours(const Grid& g, long i, long (&nb)[3][2]) {
    long rem = i, stride = 1;
    int coord[3] = {0, 0, 0};
    for (int a = g.ndim - 1; a >= 0; --a) {
        coord[a] = (int)(rem % g.n[a]);
        rem /= g.n[a];
    }
    for (int a = g.ndim - 1; a >= 0; --a) {
        const int ca = coord[a];
        const int na = g.n[a];
        long lo, hi;
        if (g.bc[a] == BC_HALO) {
            lo = (ca == 0) ? g.nc + i : i - stride;                // first layer: i < stride
            hi = (ca == na - 1) ? i + 2 * stride : i + stride;     // last layer -> nc + stride + (i - (nc - stride))
        } else if (g.bc[a] == TT_BC_PERIODIC) {
            lo = i + (long)((ca == 0) ? (na - 1) : -1) * stride;
            hi = i + (long)((ca == na - 1) ? -(na - 1) : 1) * stride;
        } else {
            const long edge = g.bc[a] == TT_BC_OUTFLOW ? i : -1;
            lo = (ca == 0) ? edge : i - stride;
            hi = (ca == na - 1) ? edge : i + stride;
        }
        nb[a][0] = lo;
        nb[a][1] = hi;
        stride *= na;
    }
}

// Quartic of Sec. 3.2 on the increasing branch T >= T_b = -(4 gamma a_r)^(-1/3):
// gamma a_r T^4 + T = rhs.  Newton from the upper bracket end; f is convex and
// increasing there, so the iterates decrease monotonically onto the root.
__device__ double t_dagger(double Tm, double Estar, double ka, double Cv, double a_r) {
    const double gamma = ka / ((1.0 + ka) * Cv);
    const double rhs = Tm + gamma * Estar;
    const double ga = gamma * a_r;
    if (ga == 0.0) return rhs;
    double T;
    if (rhs >= 0.0) {
        T = fmin(rhs, sqrt(sqrt(rhs / ga)));
    } else {
        const double Tb = -cbrt(1.0 / (4.0 * ga));
        if (rhs < 0.75 * Tb) return Tb;
        T = rhs;
    }
    for (int it = 0; it < 200; ++it) {
        const double T3 = T * T * T;
        const double f = ga * T3 * T + T - rhs;
        const double fp = 4.0 * ga * T3 + 1.0;
        const double Tn = T - f / fp;
        if (Tn == T) break;
        if (it > 0 && Tn > T) break;  // rounding floor reached (iterates stopped decreasing)
        T = Tn;
    }
    return T;
}

// Stencil coefficients of the two transport terms of every axis for cell i:
// term t of axis a is c0 X_i + cp X_{i+1} - cm X_{i-1} with c0 = w_L(i+1/2) -
// w_R(i-1/2), cp = w_R(i+1/2), cm = w_L(i-1/2) (the face weights of the flux;
// upwinding gives exactly X_i - X_{i-1} and X_{i+1} - X_i).
__device__ __forceinline__ void stencil_coefs(const Fields& f, int ndim, long i,
                                              double (&co)[3][2][3]) {
    for (int a = 0; a < ndim; ++a) {
        double lo[4], hi[4];
        if (f.fw) {
            const double* p = f.fw + (i * ndim + a) * 8;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                lo[k] = p[k];
                hi[k] = p[4 + k];
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) lo[k] = hi[k] = f.wc[k];
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            co[a][t][0] = hi[2 * t] - lo[2 * t + 1];
            co[a][t][1] = hi[2 * t + 1];
            co[a][t][2] = lo[2 * t];
        }
    }
}

// The two terms of axis a at one column (Sec. 4.3 with the ghost rows of
// Sec. 4.5): upwinding (GEN = false) takes the
// plain differences x0 - xm and xp - x0 (fewer FP64 operations, the common
// case); other fluxes the face-weighted stencil.
template <bool GEN>
__device__ __forceinline__ void axis_terms(const double (&co)[3][2][3], int a, double x0, double xm,
                                           double xp, double& t1, double& t2) {
    if (GEN) {
        t1 = co[a][0][0] * x0 + co[a][0][1] * xp - co[a][0][2] * xm;
        t2 = co[a][1][0] * x0 + co[a][1][1] * xp - co[a][1][2] * xm;
    } else {
        t1 = x0 - xm;
        t2 = xp - x0;
    }
}

// y[i][j] = X_i . thbar_j for the 1 + 2 ndim transport terms j (the grown
// quadrature vector's blocks): one lane per cell, each lane running over its
// row (consecutive columns share L1 sectors) against the block-uniform thbar.
// Because every transport term is linear in X, the quadrature of cell i's
// grown row is a combination of these dots at i and its neighbours, which
// the source stage then forms with a few scalar operations per cell.  A lane
// per cell costs nterms FMAs per element and no reduction; a warp per cell
// spent as many FP64 instructions again on the shuffle sums, and on GB300 the
// FP64 issue rate, not HBM, bounds this kernel.
__global__ void __launch_bounds__(256)
term_dots_kernel(long nrows, int nterms, int r1, const double* __restrict__ X, long ldx,
                 const double* __restrict__ thbar, double* __restrict__ y, const int* dd) {
    if (dd) {
        r1 = dd[DYN_R1];
        ldx = r1;
    }
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < nrows; i += (long)gridDim.x * blockDim.x) {
        double acc[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        const double* xi = X + i * ldx;
        for (int col = 0; col < r1; ++col) {
            const double x = xi[col];
#pragma unroll
            for (int j = 0; j < 7; ++j)
                if (j < nterms) acc[j] = fma(x, thbar[j * r1 + col], acc[j]);
        }
#pragma unroll
        for (int j = 0; j < 7; ++j)
            if (j < nterms) y[i * nterms + j] = acc[j];
    }
}

// A warp takes G <= 32 consecutive cells; lane j owns cell i0 + j for the
// scalar work.  Source stage: lane j forms its cell's E* from the term dots y
// of the cell and its neighbours (the transport terms' quadrature, Sec. 4.1
// Eq. tt_energy_density, taken through the linear stencil) and the external
// sources, then solves the quartic and forms the row scale s and the emission
// e (Sec. 3.2).  Row pass: for each cell the lanes write the scaled row, the
// scaled transport terms (the factor -s nu_a folded into one product per
// term and column), the external-source columns and the emission column.
template <bool GEN>
__global__ void __launch_bounds__(256)
transport_source_kernel(Grid g, Fields f, int transport, int source, int r1,
                        const double* __restrict__ X, long ldx, const double* __restrict__ y,
                        Sources ext, double* __restrict__ Xg, long ldg, int G, const int* dd) {
    if (dd) {  // a captured step: ranks from the device's size block
        r1 = dd[DYN_R1];
        ldx = r1;
        ldg = dd[DYN_G1];
    }
    const int lane = threadIdx.x & 31;
    const long warps = (long)gridDim.x * (blockDim.x >> 5);
    const int nterms = transport ? 1 + 2 * g.ndim : 1;
    double nu[3] = {0.0, 0.0, 0.0};
    for (int a = 0; a < g.ndim; ++a) nu[a] = f.c * f.dt / g.dx[a];
    for (long i0 = (blockIdx.x * (long)(blockDim.x >> 5) + (threadIdx.x >> 5)) * G; i0 < g.nc;
         i0 += warps * G) {
        const int cnt = (int)min((long)G, g.nc - i0);
        double scale = 1.0, emit = 0.0;
        if (source && lane < cnt) {
            const long i = i0 + lane;
            double dot = y[i * nterms];
            if (transport) {
                long nb[3][2];
                cell_neighbours(g, i, nb);
                double co[3][2][3];
                if (GEN) stencil_coefs(f, g.ndim, i, co);
                for (int a = 0; a < g.ndim; ++a) {
                    const int j1 = 1 + 2 * a, j2 = 2 + 2 * a;
                    const double m1 = nb[a][0] >= 0 ? y[nb[a][0] * nterms + j1] : 0.0;
                    const double p1 = nb[a][1] >= 0 ? y[nb[a][1] * nterms + j1] : 0.0;
                    const double m2 = nb[a][0] >= 0 ? y[nb[a][0] * nterms + j2] : 0.0;
                    const double p2 = nb[a][1] >= 0 ? y[nb[a][1] * nterms + j2] : 0.0;
                    double t1, t2, u1, u2;
                    axis_terms<GEN>(co, a, y[i * nterms + j1], m1, p1, t1, u1);
                    axis_terms<GEN>(co, a, y[i * nterms + j2], m2, p2, u2, t2);
                    dot += -nu[a] * t1 + -nu[a] * t2;
                }
            }
            // external sources: c dt x_k[i] times their quadrature q_k
            for (int k = 0; k < ext.n; ++k) dot += f.c * f.dt * ext.x[(long)k * g.nc + i] * ext.q[k];
            const double Estar = dot / f.c;
            const double ka = f.c * f.dt * f.sigma_a[i];
            const double ks = f.sigma_s ? f.c * f.dt * f.sigma_s[i] : 0.0;
            const double Td = t_dagger(f.T[i], Estar, ka, f.cv[i], f.a_r);
            const double Td2 = Td * Td;
            const double B = f.c * f.a_r * Td2 * Td2 / FOUR_PI;
            const double Jnew = (f.c * Estar / FOUR_PI + ka * B) / (1.0 + ka);
            scale = 1.0 / (1.0 + ka + ks);
            emit = scale * (ks * Jnew + ka * B);
            f.E_star[i] = Estar;
        }
        for (int j = 0; j < cnt; ++j) {
            const long i = i0 + j;
            const double sc = __shfl_sync(0xffffffffu, scale, j);
            const double em = __shfl_sync(0xffffffffu, emit, j);
            long nb[3][2];
            cell_neighbours(g, i, nb);
            double co[3][2][3];
            if (GEN) stencil_coefs(f, g.ndim, i, co);
            // term (a, t) = -s nu_a (its stencil): the factor is folded into
            // the stencil so that each output costs as few FP64 operations as
            // possible (GB300's FP64 issue rate bounds this pass): upwinding
            // writes fma(sn, xm, -sn x0) and fma(-sn, xp, sn x0), the other
            // fluxes a two-FMA chain on the scaled coefficients
            double sn[3] = {0.0, 0.0, 0.0};
            double cf[3][2][3];
            for (int a = 0; a < g.ndim; ++a) {
                sn[a] = sc * nu[a];
                if (GEN)
                    for (int t = 0; t < 2; ++t) {
                        cf[a][t][0] = -sn[a] * co[a][t][0];
                        cf[a][t][1] = -sn[a] * co[a][t][1];
                        cf[a][t][2] = sn[a] * co[a][t][2];
                    }
            }
            double* out = Xg + i * ldg;
            for (int col = lane; col < r1; col += 32) {
                const double x0 = X[i * ldx + col];
                out[col] = sc * x0;
                if (transport) {
                    for (int a = 0; a < g.ndim; ++a) {
                        const double xm = nb[a][0] >= 0 ? X[nb[a][0] * ldx + col] : 0.0;
                        const double xp = nb[a][1] >= 0 ? X[nb[a][1] * ldx + col] : 0.0;
                        if (GEN) {
                            out[(1 + 2 * a) * r1 + col] = fma(cf[a][0][0], x0, fma(cf[a][0][1], xp, cf[a][0][2] * xm));
                            out[(2 + 2 * a) * r1 + col] = fma(cf[a][1][0], x0, fma(cf[a][1][1], xp, cf[a][1][2] * xm));
                        } else {
                            const double q = sn[a] * x0;
                            out[(1 + 2 * a) * r1 + col] = fma(sn[a], xm, -q);
                            out[(2 + 2 * a) * r1 + col] = fma(-sn[a], xp, q);
                        }
                    }
                }
            }
            for (int k = lane; k < ext.n; k += 32)
                out[nterms * r1 + k] = sc * (f.c * f.dt * ext.x[(long)k * g.nc + i]);
            if (source && lane == 0) out[nterms * r1 + ext.n] = em;
        }
    }
}

// Split layout, one thread per cell: E*_i from the K spatial contractions F
// (F[i][j] = the field of term j with the angular cores integrated, before
// the spatial difference of term j is applied), then the same source stage
// as the grouped kernel (quartic, s, e); e goes to the emission block of the
// spatial core that holds it, at the cell's coordinates.
__global__ void __launch_bounds__(256)
split_source_kernel(Grid g, Fields f, StencilCo co, int transport, int K, const double* __restrict__ F,
                    double* __restrict__ eblk, long st0, long st1, long st2) {
    double nu[3] = {0.0, 0.0, 0.0};
    for (int a = 0; a < g.ndim; ++a) nu[a] = f.c * f.dt / g.dx[a];
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.nc;
         i += (long)gridDim.x * blockDim.x) {
        double dot = F[i * K];
        if (transport) {
            long nb[3][2];
            cell_neighbours(g, i, nb);
            for (int a = 0; a < g.ndim; ++a)
                for (int t = 0; t < 2; ++t) {
                    const int j = 1 + 2 * a + t;
                    const double fm = nb[a][0] >= 0 ? F[nb[a][0] * K + j] : 0.0;
                    const double fp = nb[a][1] >= 0 ? F[nb[a][1] * K + j] : 0.0;
                    dot += -nu[a] * (co.c[a][t][0] * F[i * K + j] + co.c[a][t][1] * fp - co.c[a][t][2] * fm);
                }
        }
        const double Estar = dot / f.c;
        const double ka = f.c * f.dt * f.sigma_a[i];
        const double ks = f.sigma_s ? f.c * f.dt * f.sigma_s[i] : 0.0;
        const double Td = t_dagger(f.T[i], Estar, ka, f.cv[i], f.a_r);
        const double Td2 = Td * Td;
        const double B = f.c * f.a_r * Td2 * Td2 / FOUR_PI;
        const double Jnew = (f.c * Estar / FOUR_PI + ka * B) / (1.0 + ka);
        const double sc = 1.0 / (1.0 + ka + ks);
        f.E_star[i] = Estar;
        const long c2 = i % g.n[2], q = i / g.n[2];
        const long c1 = q % g.n[1], c0 = q / g.n[1];
        eblk[c0 * st0 + c1 * st1 + c2 * st2] = sc * (ks * Jnew + ka * B);
    }
}

// HLL wave-speed factors (Sec. 3.1, after Eq. hll): for n_a >= 0,
// S_R = c n_a A(tau) and S_L = -c n_a B(tau) (mirrored for n_a < 0).
__device__ __forceinline__ double hll_A(double t, double thr) {
    if (t >= thr) return sqrt((1.0 - exp(-t * t)) / (t * t));
    return sqrt(fmax(1.0 - 0.5 * t * t, 0.0));
}
__device__ __forceinline__ double hll_B(double t, double thr) {
    if (t >= thr) return sqrt((1.0 - exp(-t * t * t * t)) / (t * t));
    return t;
}

// Face weights of Eq. hll with those speeds: F = c n^+ (w_L1 U_L + w_R1 U_R) +
// c n^- (w_L2 U_L + w_R2 U_R), w_L1 = A (1 + B) / (A + B), w_R1 = B (1 - A) / (A + B)
// and the mirror image for n < 0; tau from Eq. tauc.
__global__ void hll_weights_kernel(Grid g, const double* __restrict__ sa, const double* __restrict__ ss,
                                   double beta, double thr, double* __restrict__ fw) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.nc; i += (long)gridDim.x * blockDim.x) {
        long nb[3][2];
        cell_neighbours(g, i, nb);
        const double si = sa[i] + (ss ? ss[i] : 0.0);
        for (int a = 0; a < g.ndim; ++a) {
            for (int side = 0; side < 2; ++side) {
                const long j = nb[a][side] >= 0 ? nb[a][side] : i;
                const double sj = sa[j] + (ss ? ss[j] : 0.0);
                double tau = 0.0;
                if (si > 0.0 && sj > 0.0) tau = 2.0 * beta * g.dx[a] / (1.0 / si + 1.0 / sj);
                const double A = hll_A(tau, thr), B = hll_B(tau, thr);
                const double den = A + B;
                double* p = fw + (i * g.ndim + a) * 8 + side * 4;
                p[0] = A * (1.0 + B) / den;
                p[1] = B * (1.0 - A) / den;
                p[2] = B * (1.0 - A) / den;
                p[3] = A * (1.0 + B) / den;
            }
        }
    }
}

// Face weights of Eq. rusanov_flux_toro with S+ = c |n_a| m, m = min(1, 1 /
// tau_c) (tau_c from Eq. tauc): F = c n_a (U_L + U_R) / 2 + c |n_a| (m U_L -
// m U_R) / 2, i.e. (w_L1, w_R1, w_L2, w_R2) = (1/2, 1/2, m/2, -m/2).
__global__ void rusanov_tau_weights_kernel(Grid g, const double* __restrict__ sa, const double* __restrict__ ss,
                                           double beta, double* __restrict__ fw) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.nc; i += (long)gridDim.x * blockDim.x) {
        long nb[3][2];
        cell_neighbours(g, i, nb);
        const double si = sa[i] + (ss ? ss[i] : 0.0);
        for (int a = 0; a < g.ndim; ++a) {
            for (int side = 0; side < 2; ++side) {
                const long j = nb[a][side] >= 0 ? nb[a][side] : i;
                const double sj = sa[j] + (ss ? ss[j] : 0.0);
                double tau = 0.0;
                if (si > 0.0 && sj > 0.0) tau = 2.0 * beta * g.dx[a] / (1.0 / si + 1.0 / sj);
                const double m = tau > 1.0 ? 1.0 / tau : 1.0;
                double* p = fw + (i * g.ndim + a) * 8 + side * 4;
                p[0] = 0.5;
                p[1] = 0.5;
                p[2] = 0.5 * m;
                p[3] = -0.5 * m;
            }
        }
    }
}

__global__ void inflow_source_kernel(Grid g, Fields f, int axis, int side, int term,
                                     const double* __restrict__ gface, double* __restrict__ x) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.nc; i += (long)gridDim.x * blockDim.x) {
        long rem = i;
        int coord[3] = {0, 0, 0};
        for (int a = g.ndim - 1; a >= 0; --a) {
            coord[a] = (int)(rem % g.n[a]);
            rem /= g.n[a];
        }
        const bool on = coord[axis] == (side == 0 ? 0 : g.n[axis] - 1);
        double v = 0.0;
        if (on) {
            // face weights (w_L1, w_R1, w_L2, w_R2) of the face on this side
            double w4[4];
            if (f.fw) {
                const double* p = f.fw + (i * g.ndim + axis) * 8 + side * 4;
                for (int k = 0; k < 4; ++k) w4[k] = p[k];
            } else {
                for (int k = 0; k < 4; ++k) w4[k] = f.wc[k];
            }
            const double w = side == 0 ? w4[2 * term] : -w4[2 * term + 1];
            v = w * gface[i] / g.dx[axis];
        }
        x[i] = v;
    }
}

__global__ void __launch_bounds__(256)
energy_rows_kernel(long nc, int r, const double* __restrict__ X, long ldx,
                   const double* __restrict__ thbar, double c, double* E_out,
                   const double* __restrict__ E_star, const double* __restrict__ cv, double* T,
                   int update_T, const int* dd) {
    if (dd) {
        r = dd[DYN_R1];
        ldx = r;
    }
    // one lane per cell (see term_dots_kernel)
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < nc; i += (long)gridDim.x * blockDim.x) {
        const double* xi = X + i * ldx;
        double d0 = 0.0, d1 = 0.0;
        int col = 0;
        for (; col + 1 < r; col += 2) {
            d0 = fma(xi[col], thbar[col], d0);
            d1 = fma(xi[col + 1], thbar[col + 1], d1);
        }
        if (col < r) d0 = fma(xi[col], thbar[col], d0);
        const double E = (d0 + d1) / c;
        if (E_out) E_out[i] = E;
        if (update_T) T[i] = T[i] + (E_star[i] - E) / cv[i];
    }
}

__global__ void init_iso_kernel(long nc, const double* Tr, double c, double a_r, double* X) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < nc;
         i += (long)gridDim.x * blockDim.x) {
        const double t2 = Tr[i] * Tr[i];
        X[i] = c * a_r * t2 * t2 / FOUR_PI;
    }
}

// ------------------------------------------------------------------ adjoint
// Reverse mode of the step with the rounding's projections frozen (the
// adjoint form).  Names: Xb = adjoint of X, and so on.

// Source stage and quadrature, reversed per cell (one warp per cell): from the
// adjoint of the grown spatial core Xgb (nc x R1) and the adjoint of E* coming
// from the temperature update (Esb_in), give ybar = adjoint of the transport
// rows y (nc x nr), the rows Y themselves (for the quadrature adjoint), the
// total adjoint of E* (Esb_out), the adjoint of the input temperature (Tb_in =
// Tb_out + ...) and accumulate the sigma_a gradient.
__global__ void __launch_bounds__(256)
source_adjoint_kernel(Grid g, Fields f, int r1, const double* __restrict__ X, long ldx,
                      const double* __restrict__ thbar, const double* __restrict__ Tin,
                      const double* __restrict__ Xgb, long ldgb, const double* __restrict__ Esb_in,
                      const double* __restrict__ Tb_out, double* __restrict__ ybar,
                      double* __restrict__ Y, long ldy, double* __restrict__ Esb_out,
                      double* __restrict__ Tb_in, double* __restrict__ sigb) {
    const int lane = threadIdx.x & 31;
    const long warps = (long)gridDim.x * (blockDim.x >> 5);
    const int nterms = 1 + 2 * g.ndim;
    const int nr = nterms * r1;
    for (long i = blockIdx.x * (long)(blockDim.x >> 5) + (threadIdx.x >> 5); i < g.nc; i += warps) {
        long nb[3][2];
        cell_neighbours(g, i, nb);
        double nu[3];
        for (int a = 0; a < g.ndim; ++a) nu[a] = f.c * f.dt / g.dx[a];
        double dot = 0.0, sb = 0.0;
        const double* xg = Xgb + i * ldgb;
        for (int col = lane; col < r1; col += 32) {
            const double x0 = X[i * ldx + col];
            dot += x0 * thbar[col];
            sb += xg[col] * x0;
            for (int a = 0; a < g.ndim; ++a) {
                const double xm = nb[a][0] >= 0 ? X[nb[a][0] * ldx + col] : 0.0;
                const double xp = nb[a][1] >= 0 ? X[nb[a][1] * ldx + col] : 0.0;
                const double yp = -nu[a] * (x0 - xm), ym = -nu[a] * (xp - x0);
                dot += yp * thbar[(1 + 2 * a) * r1 + col] + ym * thbar[(2 + 2 * a) * r1 + col];
                sb += xg[(1 + 2 * a) * r1 + col] * yp + xg[(2 + 2 * a) * r1 + col] * ym;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            dot += __shfl_xor_sync(0xffffffffu, dot, o);
            sb += __shfl_xor_sync(0xffffffffu, sb, o);
        }
        const double Es = dot / f.c;
        const double ka = f.c * f.dt * f.sigma_a[i];
        const double cv = f.cv[i];
        const double Td = t_dagger(Tin[i], Es, ka, cv, f.a_r);
        const double s = 1.0 / (1.0 + ka);
        const double T3 = Td * Td * Td;
        const double B = f.c * f.a_r * T3 * Td / FOUR_PI;
        const double gamma = ka / ((1.0 + ka) * cv);
        const double fp = 4.0 * gamma * f.a_r * T3 + 1.0;
        const double eb = xg[nr];
        // e = s k B, s = 1/(1+k); B = c a_r T^4 / 4 pi; T from the quartic
        const double gB = eb * s * ka;
        double gk = eb * s * s * B - sb * s * s;
        const double gTd = gB * 4.0 * f.c * f.a_r * T3 / FOUR_PI;
        const double gEs = Esb_in[i] + gTd * gamma / fp;
        gk += gTd * (Es - f.a_r * T3 * Td) / fp * (s * s / cv);
        for (int col = lane; col < r1; col += 32) {
            const double x0 = X[i * ldx + col];
            ybar[i * ldy + col] = s * xg[col] + gEs * thbar[col] / f.c;
            Y[i * ldy + col] = x0;
            for (int a = 0; a < g.ndim; ++a) {
                const double xm = nb[a][0] >= 0 ? X[nb[a][0] * ldx + col] : 0.0;
                const double xp = nb[a][1] >= 0 ? X[nb[a][1] * ldx + col] : 0.0;
                const int cp = (1 + 2 * a) * r1 + col, cm = (2 + 2 * a) * r1 + col;
                ybar[i * ldy + cp] = s * xg[cp] + gEs * thbar[cp] / f.c;
                ybar[i * ldy + cm] = s * xg[cm] + gEs * thbar[cm] / f.c;
                Y[i * ldy + cp] = -nu[a] * (x0 - xm);
                Y[i * ldy + cm] = -nu[a] * (xp - x0);
            }
        }
        if (lane == 0) {
            Esb_out[i] = gEs;
            Tb_in[i] = Tb_out[i] + gTd / fp;
            sigb[i] += gk * f.c * f.dt;
        }
    }
}

// Transpose of the transport stencil: Xb_i from the adjoints of the rows y.
// y_j[x+] = -nu (X_j - X_lo(j)), y_j[x-] = -nu (X_hi(j) - X_j): cell i collects
// its own terms and those of the cells whose lower / upper neighbour it is.
__global__ void __launch_bounds__(256)
stencil_adjoint_kernel(Grid g, Fields f, int r1, const double* __restrict__ ybar, long ldy,
                       double* __restrict__ Xb, long ldxb) {
    const int lane = threadIdx.x & 31;
    const long warps = (long)gridDim.x * (blockDim.x >> 5);
    for (long i = blockIdx.x * (long)(blockDim.x >> 5) + (threadIdx.x >> 5); i < g.nc; i += warps) {
        long nb[3][2];
        cell_neighbours(g, i, nb);
        for (int col = lane; col < r1; col += 32) {
            double v = ybar[i * ldy + col];
            for (int a = 0; a < g.ndim; ++a) {
                const double nu = f.c * f.dt / g.dx[a];
                const int cp = (1 + 2 * a) * r1 + col, cm = (2 + 2 * a) * r1 + col;
                v += -nu * ybar[i * ldy + cp] + nu * ybar[i * ldy + cm];
                if (nb[a][1] >= 0) v += nu * ybar[nb[a][1] * ldy + cp];
                if (nb[a][0] >= 0) v -= nu * ybar[nb[a][0] * ldy + cm];
            }
            Xb[i * ldxb + col] = v;
        }
    }
}

// Grown angular cores reversed: Thb[a,l,b] += sum_j thfac_j[l] Thgb[j r1 + a, l, j r2 + b],
// Phb[b,p] += sum_j phfac_j[p] Phgb[j r2 + b, p].
__global__ void grown_theta_adjoint_kernel(int nterms, int r1, int r2, int nt, const double* Thgb,
                                           int R1, int R2, const double* tfac,
                                           double* Thb) {
    const long total = (long)r1 * nt * r2;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int b = (int)(t % r2);
        const int l = (int)((t / r2) % nt);
        const int a = (int)(t / ((long)r2 * nt));
        double v = 0.0;
        for (int j = 0; j < nterms; ++j)
            v += tfac[(long)j * nt + l] * Thgb[((long)(j * r1 + a) * nt + l) * R2 + j * r2 + b];
        Thb[t] += v;
    }
}

__global__ void grown_phi_adjoint_kernel(int nterms, int r2, int np, const double* Phgb,
                                         const double* pfac, double* Phb) {
    const long total = (long)r2 * np;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int p = (int)(t % np), b = (int)(t / np);
        double v = 0.0;
        for (int j = 0; j < nterms; ++j) v += pfac[(long)j * np + p] * Phgb[(long)(j * r2 + b) * np + p];
        Phb[t] += v;
    }
}

// Quadrature vectors reversed (thbar_j[a] = w sum_l thf_j sum_b Th[a,l,b] phibar_j[b],
// phibar_j[b] = v sum_p phf_j Ph[b,p]): given thbb (nterms x r1, scaled by sgn_j),
// add to Thb and Phb.  phibar (nterms x r2) and phibb (nterms x r2) are scratch.
__global__ void thbar_adjoint_theta_kernel(int j0, int nterms, int r1, int r2, int nt,
                                           const double* thbb, const double* phibar,
                                           const double* tfac, double w,
                                           double* Thb) {
    const long total = (long)r1 * nt * r2;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int b = (int)(t % r2);
        const int l = (int)((t / r2) % nt);
        const int a = (int)(t / ((long)r2 * nt));
        double v = 0.0;
        for (int j = j0; j < nterms; ++j)
            v += tfac[(long)j * nt + l] * thbb[j * r1 + a] * phibar[j * r2 + b];
        Thb[t] += w * v;
    }
}

// phibb[j r2 + b] = w sum_a thbb[j r1 + a] sum_l thfac_j[l] Th[a][l][b]: one warp
// per output, lanes striding over (a, l).
__global__ void thbar_adjoint_phibb_kernel(int j0, int nterms, int r1, int r2, int nt,
                                           const double* thbb, const double* Th, const double* tfac, double w, double* phibb) {
    const int lane = threadIdx.x & 31;
    const int total = nterms * r2;
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < total; t += warps) {
        const int j = t / r2, b = t % r2;
        double v = 0.0;
        if (j >= j0)
            for (int idx = lane; idx < r1 * nt; idx += 32) {
                const int a = idx / nt, l = idx - a * nt;
                v += thbb[j * r1 + a] * tfac[(long)j * nt + l] *
                     Th[((long)a * nt + l) * r2 + b];
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) phibb[t] = w * v;
    }
}

__global__ void thbar_adjoint_phi_kernel(int j0, int nterms, int r2, int np, const double* phibb,
                                         const double* pfac, double v,
                                         double* Phb) {
    const long total = (long)r2 * np;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int p = (int)(t % np), b = (int)(t / np);
        double acc = 0.0;
        for (int j = j0; j < nterms; ++j) acc += pfac[(long)j * np + p] * phibb[j * r2 + b];
        Phb[t] += v * acc;
    }
}

// Escape-energy objective on the boundary faces of vacuum axes (Sec. 4.5): for
// the high face of axis a the outward factor pair is term 1 + 2a (n_a^+), for
// the low face it is minus term 2 + 2a (-n_a^-).  Per cell: q_i = sum over its
// faces sgn dt dA_a X_i . thbar_j; Xb_i += sgn dt dA_a thbar_j.
__global__ void __launch_bounds__(256)
escape_rows_kernel(Grid g, double dt, int r, const double* __restrict__ X, long ldx,
                   const double* __restrict__ thbar_terms, double* __restrict__ qcell,
                   double* __restrict__ Xb, long ldxb, int add_grad) {
    const int lane = threadIdx.x & 31;
    const long warps = (long)gridDim.x * (blockDim.x >> 5);
    for (long i = blockIdx.x * (long)(blockDim.x >> 5) + (threadIdx.x >> 5); i < g.nc; i += warps) {
        long rem = i;
        int coord[3] = {0, 0, 0};
        for (int a = g.ndim - 1; a >= 0; --a) {
            coord[a] = (int)(rem % g.n[a]);
            rem /= g.n[a];
        }
        double q = 0.0;
        for (int a = 0; a < g.ndim; ++a) {
            if (g.bc[a] != TT_BC_VACUUM) continue;
            double dA = 1.0;
            for (int b2 = 0; b2 < g.ndim; ++b2)
                if (b2 != a) dA *= g.dx[b2];
            for (int side = 0; side < 2; ++side) {
                const bool on = side ? (coord[a] == g.n[a] - 1) : (coord[a] == 0);
                if (!on) continue;
                const int j = side ? 1 + 2 * a : 2 + 2 * a;
                const double wgt = (side ? 1.0 : -1.0) * dt * dA;
                const double* tb = thbar_terms + j * r;
                double dot = 0.0;
                for (int col = lane; col < r; col += 32) {
                    dot += X[i * ldx + col] * tb[col];
                    if (add_grad) Xb[i * ldxb + col] += wgt * tb[col];
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                q += wgt * dot;
            }
        }
        if (lane == 0) qcell[i] = q;
    }
}

// thbb_j[col] = sgn dt dA_a sum_{cells i on the face} X_i[col] (fixed order: one
// block per (face, 32-column chunk) walking the face cells sequentially).
__global__ void escape_thbb_kernel(Grid g, double dt, int r, const double* __restrict__ X, long ldx,
                                   double* __restrict__ thbb) {
    const int face = blockIdx.y;  // 2 * axis + side
    const int a = face >> 1, side = face & 1;
    const int col = blockIdx.x * 32 + threadIdx.x;
    if (a >= g.ndim || g.bc[a] != TT_BC_VACUUM || col >= r) return;
    double dA = 1.0;
    for (int b2 = 0; b2 < g.ndim; ++b2)
        if (b2 != a) dA *= g.dx[b2];
    const int j = side ? 1 + 2 * a : 2 + 2 * a;
    const double wgt = (side ? 1.0 : -1.0) * dt * dA;
    // enumerate the face cells: all coords with coord_a fixed
    const long nface = g.nc / g.n[a];
    double acc = 0.0;
    for (long t = 0; t < nface; ++t) {
        long rem = t, i = 0, stride = 1;
        for (int b2 = g.ndim - 1; b2 >= 0; --b2) {
            int cb;
            if (b2 == a) {
                cb = side ? g.n[a] - 1 : 0;
            } else {
                cb = (int)(rem % g.n[b2]);
                rem /= g.n[b2];
            }
            i += (long)cb * stride;
            stride *= g.n[b2];
        }
        acc += X[i * ldx + col];
    }
    thbb[j * r + col] = wgt * acc;
}

__global__ void energy_adjoint_kernel(long nc, int r, const double* __restrict__ thbar, double c,
                                      const double* __restrict__ cv, const double* __restrict__ Tb,
                                      double* __restrict__ Xb, long ldxb, double* __restrict__ e1b,
                                      double* __restrict__ Esb) {
    const int lane = threadIdx.x & 31;
    const long warps = (long)gridDim.x * (blockDim.x >> 5);
    for (long i = blockIdx.x * (long)(blockDim.x >> 5) + (threadIdx.x >> 5); i < nc; i += warps) {
        const double E1b = -Tb[i] / cv[i];
        for (int col = lane; col < r; col += 32) Xb[i * ldxb + col] += E1b * thbar[col] / c;
        if (lane == 0) {
            e1b[i] = E1b / c;
            Esb[i] = Tb[i] / cv[i];
        }
    }
}

__global__ void sum_kernel(long n, const double* x, double* out) {
    __shared__ double sh[256];
    double a = 0.0;
    for (long i = threadIdx.x; i < n; i += blockDim.x) a += x[i];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out += sh[0];
}

constexpr int RED_BLOCKS = 1024;

__global__ void totals_partial_kernel(long nc, const double* E, const double* cv, const double* T,
                                      double* part) {
    __shared__ double s0[256], s1[256];
    double a = 0.0, b = 0.0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < nc;
         i += (long)gridDim.x * blockDim.x) {
        a += E[i];
        b += cv[i] * T[i];
    }
    s0[threadIdx.x] = a;
    s1[threadIdx.x] = b;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            s0[threadIdx.x] += s0[threadIdx.x + o];
            s1[threadIdx.x] += s1[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[blockIdx.x] = s0[0];
        part[RED_BLOCKS + blockIdx.x] = s1[0];
    }
}

// The partials summed in a fixed tree (one thread's chain of 2048 additions took
// 105 us on GB300, the tree 5).
__global__ void __launch_bounds__(256) totals_final_kernel(const double* part, double* totals) {
    __shared__ double s_a[8], s_b[8];
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < RED_BLOCKS; k += 256) {
        a += part[k];
        b += part[RED_BLOCKS + k];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s_a[threadIdx.x >> 5] = a;
        s_b[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            a += s_a[w];
            b += s_b[w];
        }
        totals[0] = a;
        totals[1] = b;
    }
}

inline int blocks_for(long total, int threads = 256) {
    long b = (total + threads - 1) / threads;
    return (int)std::max<long>(1, std::min<long>(b, 152L * 32));
}

}  // namespace

void build_grown_angular(cudaStream_t s, const Angular& ang, int ndim, bool transport,
                         bool source, int r1, int r2, const double* Th, const double* Ph,
                         double* Thg, double* Phg, int R1, int R2, const Sources& ext, const int* dd) {
    const int nterms = transport ? 1 + 2 * ndim : 1;
    note_launch();
    grown_theta_kernel<<<blocks_for((long)R1 * ang.n_theta * R2), 256, 0, s>>>(
        nterms, source ? 1 : 0, r1, r2, ang.n_theta, Th, ang.tfac, ext.n, ext.th, Thg,
        R1, R2, dd);
    note_launch();
    grown_phi_kernel<<<blocks_for((long)R2 * ang.n_phi), 256, 0, s>>>(
        nterms, source ? 1 : 0, r2, ang.n_phi, Ph, ang.pfac, ext.n, ext.ph, Phg, R2, dd);
}

// phibar scratch: thbar + nterms*r1 (caller allocates (nterms*(r1+r2)) doubles at thbar)
void grown_thbar(cudaStream_t s, const Angular& ang, int ndim, bool transport, int r1, int r2,
                 const double* Th, const double* Ph, double* thbar, const int* dd) {
    const int nterms = transport ? 1 + 2 * ndim : 1;
    double* phibar = thbar + nterms * r1;
    note_launch();
    phibar_kernel<<<blocks_for((long)nterms * r2), 256, 0, s>>>(nterms, r2, ang.n_phi, Ph,
                                                               ang.pfac, ang.v, phibar, dd);
    note_launch();
    thbar_kernel<<<blocks_for((long)nterms * r1 * 32, 128), 128, 0, s>>>(
        nterms, r1, r2, ang.n_theta, Th, ang.tfac, ang.w, phibar, thbar, dd);
}

void plain_thbar(cudaStream_t s, const Angular& ang, int r1, int r2, const double* Th,
                 const double* Ph, double* thbar, const int* dd) {
    grown_thbar(s, ang, 0, false, r1, r2, Th, Ph, thbar, dd);
}

void transport_source_rows(cudaStream_t s, const Grid& g, const Fields& f, bool transport,
                           bool source, int r1, const double* X, long ldx, const double* thbar,
                           double* Xg, long ldg, double* ydots, const Sources& ext, const int* dd) {
    const int nterms = transport ? 1 + 2 * g.ndim : 1;
    if (source) {
        // a shard's stencil also reads the dots of its two halo layers (rows
        // nc .. nc + 2 stride - 1, BC_HALO on axis 0)
        const long ny = g.nc + (transport && g.bc[0] == BC_HALO ? 2 * (g.nc / g.n[0]) : 0);
        const int yb = (int)std::max<long>(1, std::min<long>((ny + 255) / 256, 152L * 8));
        note_launch();
        term_dots_kernel<<<yb, 256, 0, s>>>(ny, nterms, r1, X, ldx, thbar, ydots, dd);
    }
    // cells per warp: up to 32 (the scalar source stage then fills every lane),
    // fewer on small grids so that about 32 warps per SM stay busy
    const int G = (int)std::max<long>(1, std::min<long>(32, g.nc / (152L * 32)));
    const long warps_needed = (g.nc + G - 1) / G;
    const int blocks = (int)std::max<long>(1, std::min<long>((warps_needed + 7) / 8, 152L * 64));
    note_launch();
    if (f.flux == TT_FLUX_UPWIND)
        transport_source_kernel<false><<<blocks, 256, 0, s>>>(g, f, transport ? 1 : 0, source ? 1 : 0, r1,
                                                              X, ldx, ydots, ext, Xg, ldg, G, dd);
    else
        transport_source_kernel<true><<<blocks, 256, 0, s>>>(g, f, transport ? 1 : 0, source ? 1 : 0, r1,
                                                             X, ldx, ydots, ext, Xg, ldg, G, dd);
}

void energy_rows(cudaStream_t s, long nc, int r, const double* X, long ldx, const double* thbar,
                 double c, double* E_out, const double* E_star, const double* cv, double* T,
                 bool update_T, const int* dd) {
    const int blocks = (int)std::max<long>(1, std::min<long>((nc + 255) / 256, 152L * 8));
    note_launch();
    energy_rows_kernel<<<blocks, 256, 0, s>>>(nc, r, X, ldx, thbar, c, E_out, E_star, cv, T,
                                              update_T ? 1 : 0, dd);
}

void split_source_cells(cudaStream_t s, const Grid& g, const Fields& f, const StencilCo& co,
                        bool transport, int K, const double* F, double* eblk, long st0, long st1,
                        long st2) {
    note_launch();
    split_source_kernel<<<blocks_for(g.nc), 256, 0, s>>>(g, f, co, transport ? 1 : 0, K, F, eblk, st0,
                                                        st1, st2);
}

void hll_face_weights(cudaStream_t s, const Grid& g, const double* sigma_a, const double* sigma_s,
                      double beta, double tau_threshold, double* fw) {
    note_launch();
    hll_weights_kernel<<<blocks_for(g.nc), 256, 0, s>>>(g, sigma_a, sigma_s, beta, tau_threshold, fw);
}

void rusanov_tau_face_weights(cudaStream_t s, const Grid& g, const double* sigma_a, const double* sigma_s,
                              double beta, double* fw) {
    note_launch();
    rusanov_tau_weights_kernel<<<blocks_for(g.nc), 256, 0, s>>>(g, sigma_a, sigma_s, beta, fw);
}

void inflow_source(cudaStream_t s, const Grid& g, const Fields& f, int axis, int side, int term,
                   const double* gface, double* x) {
    note_launch();
    inflow_source_kernel<<<blocks_for(g.nc), 256, 0, s>>>(g, f, axis, side, term, gface, x);
}

void init_isotropic(cudaStream_t s, long nc, const double* Tr, double c, double a_r, double* X) {
    note_launch();
    init_iso_kernel<<<blocks_for(nc), 256, 0, s>>>(nc, Tr, c, a_r, X);
}

void source_adjoint_rows(cudaStream_t s, const Grid& g, const Fields& f, int r1, const double* X,
                         long ldx, const double* thbar, const double* Tin, const double* Xgb,
                         long ldgb, const double* Esb_in, const double* Tb_out, double* ybar,
                         double* Y, long ldy, double* Esb_out, double* Tb_in, double* sigb) {
    const int blocks = (int)std::max<long>(1, std::min<long>((g.nc + 7) / 8, 152L * 64));
    note_launch();
    source_adjoint_kernel<<<blocks, 256, 0, s>>>(g, f, r1, X, ldx, thbar, Tin, Xgb, ldgb, Esb_in,
                                                 Tb_out, ybar, Y, ldy, Esb_out, Tb_in, sigb);
}

void stencil_adjoint_rows(cudaStream_t s, const Grid& g, const Fields& f, int r1, const double* ybar,
                          long ldy, double* Xb, long ldxb) {
    const int blocks = (int)std::max<long>(1, std::min<long>((g.nc + 7) / 8, 152L * 64));
    note_launch();
    stencil_adjoint_kernel<<<blocks, 256, 0, s>>>(g, f, r1, ybar, ldy, Xb, ldxb);
}

void grown_angular_adjoint(cudaStream_t s, const Angular& ang, int ndim, int r1, int r2,
                           const double* Thgb, const double* Phgb, int R1, int R2, double* Thb,
                           double* Phb) {
    const int nterms = 1 + 2 * ndim;
    note_launch();
    grown_theta_adjoint_kernel<<<blocks_for((long)r1 * ang.n_theta * r2), 256, 0, s>>>(
        nterms, r1, r2, ang.n_theta, Thgb, R1, R2, ang.tfac, Thb);
    note_launch();
    grown_phi_adjoint_kernel<<<blocks_for((long)r2 * ang.n_phi), 256, 0, s>>>(
        nterms, r2, ang.n_phi, Phgb, ang.pfac, Phb);
}

void thbar_adjoint(cudaStream_t s, const Angular& ang, int nterms, int j0, int r1, int r2,
                   const double* Th, const double* Ph, const double* thbb, double* scratch,
                   double* Thb, double* Phb) {
    double* phibar = scratch;                 // nterms * r2
    double* phibb = scratch + nterms * r2;    // nterms * r2
    note_launch();
    phibar_kernel<<<blocks_for((long)nterms * r2), 256, 0, s>>>(nterms, r2, ang.n_phi, Ph, ang.pfac, ang.v, phibar,
                                                               nullptr);
    note_launch();
    thbar_adjoint_theta_kernel<<<blocks_for((long)r1 * ang.n_theta * r2), 256, 0, s>>>(
        j0, nterms, r1, r2, ang.n_theta, thbb, phibar, ang.tfac, ang.w, Thb);
    note_launch();
    thbar_adjoint_phibb_kernel<<<blocks_for((long)nterms * r2 * 32, 128), 128, 0, s>>>(
        j0, nterms, r1, r2, ang.n_theta, thbb, Th, ang.tfac, ang.w, phibb);
    note_launch();
    thbar_adjoint_phi_kernel<<<blocks_for((long)r2 * ang.n_phi), 256, 0, s>>>(
        j0, nterms, r2, ang.n_phi, phibb, ang.pfac, ang.v, Phb);
}

void escape_rows(cudaStream_t s, const Grid& g, double dt, int r, const double* X, long ldx,
                 const double* thbar_terms, double* qcell, double* Xb, long ldxb, bool add_grad) {
    const int blocks = (int)std::max<long>(1, std::min<long>((g.nc + 7) / 8, 152L * 64));
    note_launch();
    escape_rows_kernel<<<blocks, 256, 0, s>>>(g, dt, r, X, ldx, thbar_terms, qcell, Xb, ldxb,
                                              add_grad ? 1 : 0);
}

void escape_thbb(cudaStream_t s, const Grid& g, double dt, int r, const double* X, long ldx,
                 double* thbb) {
    note_launch();
    escape_thbb_kernel<<<dim3((r + 31) / 32, 6), 32, 0, s>>>(g, dt, r, X, ldx, thbb);
}

void energy_adjoint_rows(cudaStream_t s, long nc, int r, const double* thbar, double c,
                         const double* cv, const double* Tb, double* Xb, long ldxb, double* e1b,
                         double* Esb) {
    const int blocks = (int)std::max<long>(1, std::min<long>((nc + 7) / 8, 152L * 64));
    note_launch();
    energy_adjoint_kernel<<<blocks, 256, 0, s>>>(nc, r, thbar, c, cv, Tb, Xb, ldxb, e1b, Esb);
}

void sum_into(cudaStream_t s, long n, const double* x, double* out) {
    note_launch();
    sum_kernel<<<1, 256, 0, s>>>(n, x, out);
}

void energy_totals(cudaStream_t s, long nc, const double* E, const double* cv, const double* T,
                   double* totals_dev, double* scratch) {
    note_launch();
    totals_partial_kernel<<<RED_BLOCKS, 256, 0, s>>>(nc, E, cv, T, scratch);
    note_launch();
    totals_final_kernel<<<1, 256, 0, s>>>(scratch, totals_dev);
}

}  // namespace ttsn
