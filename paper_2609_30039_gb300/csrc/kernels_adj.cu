// Transposed (discrete-adjoint) half-steps, arxiv 2609.30039 Sec. 3.1, Eq. (adjoint).
//
// Every forward update has a transpose kernel of the same locality, in a general form (CPML,
// PEC, poles: k_adj_e_gen / k_adj_h_gen) and an interior form (k_adj_e_int / k_adj_h_int):
//   * k_adj_e*  (one thread per E column, like the forward E update) applies the transpose of
//     the forward H update (Ebar += gathered backward differences of the H cotangent, the
//     opposite-direction differences of Sec. 3.1), injects dJ/dE of the monitors, and
//     transposes the E update's own-cell part (poles, eps^-1, material cotangent);
//   * k_adj_h*  (one thread per H column) applies the transpose of the forward E update
//     (Hbar += gathered forward differences) and the H-side CPML recursion.
// CPML transpose (Sec. 3.1): psibar_mem = psibar + ybar, Dbar = ybar/kappa + c psibar_mem,
// psibar_old = b psibar_mem.  Pole transpose: the 2x2 trapezoidal system applied to the
// cotangents with M^T.
//
// Gather form needs the cotangent of every neighbour's derivative D while its owner is still
// updating psibar.  So that no kernel reads a value another thread of the same launch writes,
// the E-side own-cell part of transposed step m is deferred to the next k_adj_e* (m-1):
// after k_adj_e*(m) the E array holds F = S/(eps_inf + G) * Etilde_bar (the cotangent of the
// curl, which k_adj_h needs at neighbours), and the pole/psi cotangents still hold their step
// m+1 values.  k_adj_e*(m-1) (or k_adj_flush) first completes step m for its own cell:
//   Ebar^m   = (eps_inf - G)/S * F + sum_p g_p . xbar_p
//   xbar_p^m = M_p^T xbar_p + ((1 - M00_p) / S, -M01_p / S) F
//   psibar_E^m = b (psibar_E + (+F | -F))
// The H side needs no deferral: psibar_H of step m is finished by k_adj_h*(m) after
// k_adj_e*(m) has read it.
#include <algorithm>

#include "fdtd_internal.cuh"

namespace gbfdtd {

// Completes the deferred own-cell transpose of an E update for component a; returns Ebar.
template <typename T>
__device__ __forceinline__ T e_deferred(const Dom<T>& d, int a, int i, int j, int k, long long id, bool disp,
                                        T F, T S) {
    const int c[3] = {i, j, k};
    const T ie = d.ie[a][id];
    T eb;
    if (disp) {
        eb = (T(1) / ie - d.G) / S * F;
        const long long bo = ade_off(d, i, j, k);
        for (int p = 0; p < d.npole; ++p) {
            T* pp = d.aade + ((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo;
            T* pq = d.aade + ((long long)(a * d.npole + p) * 2 + 1) * d.bcell + bo;
            const T xp = *pp, xq = *pq;
            eb += d.g0[p] * xp + d.g1[p] * xq;
            *pp = d.M00[p] * xp + d.M10[p] * xq + (T(1) - d.M00[p]) / S * F;
            *pq = d.M01[p] * xp + d.M11[p] * xq - d.M01[p] / S * F;
        }
    } else {
        eb = F / (S * ie);
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int ax = (a + 1 + s) % 3;
        if (d.ns[ax] == 0) continue;
        const int x = c[ax];
        const int sl = slab_of(x, d.dlo[ax], d.dhi[ax], d.n[ax]);
        if (sl < 0) continue;
        T* p = d.apsiE[a][s] + slab_off(d.n, d.ns, ax, i, j, k, sl);
        *p = d.cE[ax][x] * (*p + (s == 0 ? F : -F));
    }
    return eb;
}

template <typename T>
__device__ __forceinline__ double inject_at(const Dom<T>& d, const Mon* __restrict__ mons, int comp, int i, int j,
                                            int k, long long pidx) {
    // dJ/df(t) = Re(conj(cot) exp(i w t)), pidx = (step * 2 + kind) of the phase table
    double acc = 0.0;
    for (int mm = 0; mm < d.nmon; ++mm) {
        const Mon& m = mons[d.mon[mm]];
        if (!m.cot || !((m.mask >> comp) & 1u)) continue;
        if (i < m.lo[0] || i >= m.hi[0] || j < m.lo[1] || j >= m.hi[1] || k < m.lo[2] || k >= m.hi[2]) continue;
        int ci = 0;
        for (int c2 = 0; c2 < comp; ++c2) ci += (m.mask >> c2) & 1u;
        const long long cell = ((long long)(k - m.lo[2]) * m.by + (j - m.lo[1])) * m.bx + (i - m.lo[0]);
        const double2* ph = m.phase + pidx * m.nf;
        const double2* ct = m.cot + (long long)ci * m.nf * m.ncell + cell;
        for (int f = 0; f < m.nf; ++f) {
            const double2 c = ct[(long long)f * m.ncell];
            const double2 p = ph[f];
            acc += c.x * p.x + c.y * p.y;
        }
    }
    return acc;
}

// ---- general tiles, hoisted form -------------------------------------------------------------
// Column constants (CPML coefficients along x and y at this column and its -1 / +1 neighbour)
// are computed once per thread; along z once per plane.  Per plane every load precedes every
// store.  The cotangent terms of the z-derivatives are carried from plane to plane.

template <typename T>
struct CpmlC {   // coefficients of one node: slab index (-1 outside), b, c, 1/kappa
    int s;
    T b, c, k;
};

template <typename T>
__device__ __forceinline__ CpmlC<T> cpml_c(const Dom<T>& d, const T* coef, int q, int x) {
    CpmlC<T> r;
    r.s = (d.ns[q] && x >= 0 && x < d.n[q]) ? slab_of(x, d.dlo[q], d.dhi[q], d.n[q]) : -1;
    r.b = T(1);
    r.c = T(0);
    r.k = T(1);
    if (r.s >= 0) {
        const int N = d.n[q];
        r.b = coef[x];
        r.c = coef[N + x];
        r.k = coef[2 * N + x];
    }
    return r;
}

// Dbar of a derivative whose ybar is yb, at a node with coefficients cc and memory cotangent ps.
template <typename T>
__device__ __forceinline__ T dbar_c(const CpmlC<T>& cc, T yb, T ps) {
    return cc.s >= 0 ? cc.k * yb + cc.c * (ps + yb) : yb;
}

// Offsets of a cell inside the slab arrays of each axis.
template <typename T>
__device__ __forceinline__ long long off_x(const Dom<T>& d, int s, int j, int k) {
    return ((long long)k * d.n[1] + j) * d.ns[0] + s;
}
template <typename T>
__device__ __forceinline__ long long off_y(const Dom<T>& d, int s, int i, int k) {
    return ((long long)k * d.ns[1] + s) * d.n[0] + i;
}
template <typename T>
__device__ __forceinline__ long long off_z(const Dom<T>& d, int s, int i, int j) {
    return ((long long)s * d.n[1] + j) * d.n[0] + i;
}

// Transposed E step of column (i, j) over planes [z0, z1) in general form (CPML, PEC, poles,
// periodic wrap); `flags` tells whether monitor injection can apply.  pacc (or nullptr): this
// thread's sums of the pole-coefficient cotangents [pole][M00, M01, M10, M11, g0, g1].
template <typename T>
__device__ __forceinline__ void adj_e_column(const Dom<T>& d, const Mon* __restrict__ mons, int i, int j, int z0,
                                             int z1, int flags, T S, int m, int pending, double* pacc) {
    const int nx = d.n[0], ny = d.n[1];
    const long long nxy = (long long)nx * ny;
    T* A0 = d.A[0];
    T* A1 = d.A[1];
    T* A2 = d.A[2];
    const T* B0 = d.A[3];
    const T* B1 = d.A[4];
    const T* B2 = d.A[5];
    // E-node coefficients (deferred psibar_E), H-node coefficients at this column and the -1 one
    const CpmlC<T> xE = cpml_c(d, d.cE[0], 0, i), yE = cpml_c(d, d.cE[1], 1, j);
    const CpmlC<T> xH = cpml_c(d, d.cH[0], 0, i), xHm = cpml_c(d, d.cH[0], 0, i - 1);
    const CpmlC<T> yH = cpml_c(d, d.cH[1], 1, j), yHm = cpml_c(d, d.cH[1], 1, j - 1);
    const bool pi = i == 0 && !d.per[0], pj = j == 0 && !d.per[1];   // PEC plane at this column
    bool hasx, hasy;                                                   // -x / -y neighbour exists
    const long long oxm = nb_minus(i, nx, 1, d.per[0], &hasx);
    const long long oym = nb_minus(j, ny, nx, d.per[1], &hasy);
    const bool gcol = d.design && i >= d.glo[0] && i < d.ghi[0] && j >= d.glo[1] && j < d.ghi[1];
    const bool mon = d.nmon && (flags & kTileMonE);
    long long id = (long long)z0 * nxy + (long long)j * nx + i;
    // z-derivative terms of H_y (s = 0) and H_x (s = 1) at plane k-1
    T tyz_m = T(0), txz_m = T(0);
    if (z0 > 0) {
        const CpmlC<T> zH = cpml_c(d, d.cH[2], 2, z0 - 1);
        const long long o = zH.s >= 0 ? off_z(d, zH.s, i, j) : 0;
        tyz_m = dbar_c(zH, -S * B1[id - nxy], zH.s >= 0 ? d.apsiH[1][0][o] : T(0));
        txz_m = dbar_c(zH, S * B0[id - nxy], zH.s >= 0 ? d.apsiH[0][1][o] : T(0));
    }
    for (int k = z0; k < z1; ++k, id += nxy) {
        const bool pk = k == 0;
        const bool px = pj || pk, py = pi || pk, pz = pi || pj;
        const CpmlC<T> zE = cpml_c(d, d.cE[2], 2, k), zH = cpml_c(d, d.cH[2], 2, k);
        // loads of the plane
        const T f0 = A0[id], f1 = A1[id], f2 = A2[id];
        const T b0 = B0[id], b1 = B1[id], b2 = B2[id];
        const T b2_xm = hasx ? B2[id + oxm] : T(0), b1_xm = hasx ? B1[id + oxm] : T(0);
        const T b2_ym = hasy ? B2[id + oym] : T(0), b0_ym = hasy ? B0[id + oym] : T(0);
        const long long oz = zH.s >= 0 ? off_z(d, zH.s, i, j) : 0;
        const T p10 = zH.s >= 0 ? d.apsiH[1][0][oz] : T(0);   // H_y, d/dz
        const T p01 = zH.s >= 0 ? d.apsiH[0][1][oz] : T(0);   // H_x, d/dz
        const T p20 = xH.s >= 0 ? d.apsiH[2][0][off_x(d, xH.s, j, k)] : T(0);                 // H_z, d/dx
        const T p20m = (hasx && xHm.s >= 0) ? d.apsiH[2][0][off_x(d, xHm.s, j, k)] : T(0);
        const T p11 = xH.s >= 0 ? d.apsiH[1][1][off_x(d, xH.s, j, k)] : T(0);                 // H_y, d/dx
        const T p11m = (hasx && xHm.s >= 0) ? d.apsiH[1][1][off_x(d, xHm.s, j, k)] : T(0);
        const T p21 = yH.s >= 0 ? d.apsiH[2][1][off_y(d, yH.s, i, k)] : T(0);                 // H_z, d/dy
        const T p21m = (hasy && yHm.s >= 0) ? d.apsiH[2][1][off_y(d, yHm.s, i, k)] : T(0);
        const T p00 = yH.s >= 0 ? d.apsiH[0][0][off_y(d, yH.s, i, k)] : T(0);                 // H_x, d/dy
        const T p00m = (hasy && yHm.s >= 0) ? d.apsiH[0][0][off_y(d, yHm.s, i, k)] : T(0);
        // derivative cotangents of the H update: s = 0 has ybar = -S Hbar, s = 1 has +S Hbar
        const T tyz = dbar_c(zH, -S * b1, p10), txz = dbar_c(zH, S * b0, p01);
        const T tzx = dbar_c(xH, -S * b2, p20), tzx_m = hasx ? dbar_c(xHm, -S * b2_xm, p20m) : T(0);
        const T tyx = dbar_c(xH, S * b1, p11), tyx_m = hasx ? dbar_c(xHm, S * b1_xm, p11m) : T(0);
        const T tzy = dbar_c(yH, S * b2, p21), tzy_m = hasy ? dbar_c(yHm, S * b2_ym, p21m) : T(0);
        const T txy = dbar_c(yH, -S * b0, p00), txy_m = hasy ? dbar_c(yHm, -S * b0_ym, p00m) : T(0);
        const bool dcell = d.npole > 0 && i >= d.blo[0] && i < d.bhi[0] && j >= d.blo[1] && j < d.bhi[1] &&
                           k >= d.blo[2] && k < d.bhi[2] && d.mask[id];
        const bool gcell = gcol && k >= d.glo[2] && k < d.ghi[2];
        const T fin[3] = {f0, f1, f2};
        const T gat[3] = {(tyz_m - tyz) + (tzy_m - tzy), (tzx_m - tzx) + (txz_m - txz), (txy_m - txy) + (tyx_m - tyx)};
        const bool pec[3] = {px, py, pz};
        // own-cell CPML nodes of E_a's two derivatives (s = 0 along (a+1)%3, s = 1 along (a+2)%3)
        const CpmlC<T>* ec[3][2] = {{&yE, &zE}, {&zE, &xE}, {&xE, &yE}};
        T fout[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (pec[a]) {
                fout[a] = T(0);
                continue;
            }
            const T ie = d.ie[a][id];
            const T F = fin[a];
            T eb;
            if (pending) {
                // complete the own-cell transpose of step m+1
                if (dcell) {
                    eb = (T(1) / ie - d.G) / S * F;
                    const long long bo = ade_off(d, i, j, k);
                    for (int p = 0; p < d.npole; ++p) {
                        T* pp = d.aade + ((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo;
                        T* pq = d.aade + ((long long)(a * d.npole + p) * 2 + 1) * d.bcell + bo;
                        const T xp = *pp, xq = *pq;
                        eb += d.g0[p] * xp + d.g1[p] * xq;
                        *pp = d.M00[p] * xp + d.M10[p] * xq + (T(1) - d.M00[p]) / S * F;
                        *pq = d.M01[p] * xp + d.M11[p] * xq - d.M01[p] / S * F;
                    }
                } else {
                    eb = F / (S * ie);
                }
#pragma unroll
                for (int s2 = 0; s2 < 2; ++s2) {
                    const CpmlC<T>& cc = *ec[a][s2];
                    if (cc.s < 0) continue;
                    const int ax = (a + 1 + s2) % 3;
                    const long long o = ax == 0 ? off_x(d, cc.s, j, k) : (ax == 1 ? off_y(d, cc.s, i, k) : off_z(d, cc.s, i, j));
                    T* pp = d.apsiE[a][s2] + o;
                    *pp = cc.b * (*pp + (s2 == 0 ? F : -F));
                }
            } else {
                eb = F;
            }
            eb += gat[a];
            if (mon) eb += (T)inject_at(d, mons, a, i, j, k, (long long)m * 2 + 0);
            T et = eb;
            T gdisp = T(0);
            if (dcell) {
                const long long bo = ade_off(d, i, j, k);
                for (int p = 0; p < d.npole; ++p) {
                    const T xp = d.aade[((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo];
                    const T xq = d.aade[((long long)(a * d.npole + p) * 2 + 1) * d.bcell + bo];
                    et += d.g0[p] * xp + d.g1[p] * xq;
                }
                gdisp = d.G;
            }
            const bool pcell = pacc && dcell;
            if (gcell || pcell) {
                const int b = (a + 1) % 3, q = (a + 2) % 3;
                // -1 neighbours along b and q (this component is not PEC-held, so they exist,
                // wrapping on a periodic axis); the cell lies outside the CPML slabs, so the
                // forward update used the plain curl
                const long long om[3] = {oxm, oym, -nxy};
                const T* Hq = d.F[3 + q];
                const T* Hb = d.F[3 + b];
                const T curl = (Hq[id] - Hq[id + om[b]]) - (Hb[id] - Hb[id + om[q]]);
                double delta = (double)(S * curl);
                const T e0 = d.F[a][id];
                const long long bo = dcell ? ade_off(d, i, j, k) : 0;
                if (dcell) {
                    for (int p = 0; p < d.npole; ++p) {
                        const T P = d.ade[((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo];
                        const T Q = d.ade[((long long)(a * d.npole + p) * 2 + 1) * d.bcell + bo];
                        delta += (double)(P - (d.M00[p] * P + d.M01[p] * Q) - T(2) * d.g0[p] * e0);
                    }
                }
                // E^{m+1} = E^m + rho delta with rho = eps^-1 / (1 + eps^-1 G)
                const double r = 1.0 / (1.0 + (double)ie * (double)gdisp);
                if (gcell) {
                    const long long gi = ((long long)(k - d.glo[2]) * (d.ghi[1] - d.glo[1]) + (j - d.glo[1])) *
                                             (d.ghi[0] - d.glo[0]) + (i - d.glo[0]);
                    const long long gn =
                        (long long)(d.ghi[0] - d.glo[0]) * (d.ghi[1] - d.glo[1]) * (d.ghi[2] - d.glo[2]);
                    d.grad[a * gn + gi] += (double)et * delta * r * r;
                }
                if (pcell) {
                    // x_p^{m+1} = M_p x_p^m + g_p es with es = E^m + E^{m+1}; E^{m+1} depends on
                    // M00, M01 (through delta) and on g0 (through delta and G): with et the total
                    // cotangent of E^{m+1} and u = xbar_P - rho et,
                    //   M00 += u P, M01 += u Q, M10 += xbar_Q P, M11 += xbar_Q Q,
                    //   g0 += u es,  g1 += xbar_Q es
                    const double rho = (double)ie * r;
                    const double es = 2.0 * (double)e0 + rho * delta;
                    const double etr = (double)et * rho;
                    for (int p = 0; p < d.npole; ++p) {
                        const long long o0 = ((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo;
                        const long long o1 = o0 + d.bcell;
                        const double P = (double)d.ade[o0], Q = (double)d.ade[o1];
                        const double xq = (double)d.aade[o1];
                        const double u = (double)d.aade[o0] - etr;
                        double* pa = pacc + 6 * p;
                        pa[0] += u * P;
                        pa[1] += u * Q;
                        pa[2] += xq * P;
                        pa[3] += xq * Q;
                        pa[4] += u * es;
                        pa[5] += xq * es;
                    }
                }
            }
            fout[a] = S * ie / (T(1) + ie * gdisp) * et;
        }
        A0[id] = fout[0];
        A1[id] = fout[1];
        A2[id] = fout[2];
        tyz_m = tyz;
        txz_m = txz;
    }
}

// kPG: also sums the pole-coefficient cotangents of domains that collect them (Sec. 3.1: pole
// parameters through the transposed dispersion update): per thread over its column, then one
// warp sum and one FP64 atomic per warp and coefficient into the domain's accumulator.
template <typename T, bool kPG>
__global__ void __launch_bounds__(kTileX* kTileY, sizeof(T) == 4 ? 3 : 2)
    k_adj_e_gen(const Dom<T>* __restrict__ doms, const Mon* __restrict__ mons, const Tile* __restrict__ tiles, T S,
                int m, int pending) {
    const Tile t = tiles[blockIdx.x];
    int i, j;
    tile_coords(t, i, j);
    const Dom<T>& d = doms[t.dom];
    if (!kPG) {
        if (i < 0 || j < 0) return;
        adj_e_column(d, mons, i, j, t.z0, t.z1, t.flags, S, m, pending, (double*)nullptr);
        return;
    }
    // every lane of a warp reaches the shuffles below (the domain, hence np, is the block's)
    const int np = d.pgc ? d.npole : 0;
    double acc[kMaxPole * 6];
    for (int q = 0; q < np * 6; ++q) acc[q] = 0.0;
    if (i >= 0 && j >= 0) adj_e_column(d, mons, i, j, t.z0, t.z1, t.flags, S, m, pending, np ? acc : nullptr);
    for (int q = 0; q < np * 6; ++q) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(d.pgc + q, v);
    }
}

// Transposed H step of column (i, j) over planes [z0, z1) in general form.
template <typename T>
__device__ __forceinline__ void adj_h_column(const Dom<T>& d, const Mon* __restrict__ mons, int i, int j, int z0,
                                             int z1, int flags, T S, int m) {
    const int nx = d.n[0], ny = d.n[1], nz = d.n[2];
    const long long nxy = (long long)nx * ny;
    const T* A0 = d.A[0];
    const T* A1 = d.A[1];
    const T* A2 = d.A[2];
    T* B0 = d.A[3];
    T* B1 = d.A[4];
    T* B2 = d.A[5];
    bool xe, ye;   // the +x / +y neighbour exists (wraps on a periodic axis)
    const long long oxp = nb_plus(i, nx, 1, d.per[0], &xe);
    const long long oyp = nb_plus(j, ny, nx, d.per[1], &ye);
    const bool pi = i == 0 && !d.per[0], pj = j == 0 && !d.per[1];   // PEC plane at this column
    // H-node coefficients (own psibar_H); E-node coefficients at this column and the +1 one
    const CpmlC<T> xH = cpml_c(d, d.cH[0], 0, i), yH = cpml_c(d, d.cH[1], 1, j);
    const CpmlC<T> xE = cpml_c(d, d.cE[0], 0, i), xEp = cpml_c(d, d.cE[0], 0, i + 1);
    const CpmlC<T> yE = cpml_c(d, d.cE[1], 1, j), yEp = cpml_c(d, d.cE[1], 1, j + 1);
    const bool mon = d.nmon && m >= 1 && (flags & kTileMonH);
    long long id = (long long)z0 * nxy + (long long)j * nx + i;
    // z-derivative terms of E_y (s = 0) and E_x (s = 1) at plane k (carried to the next plane)
    auto zterms = [&](int k, long long idk, T& ty, T& tx) {
        if (k >= nz) {
            ty = T(0);
            tx = T(0);
            return;
        }
        const CpmlC<T> zE = cpml_c(d, d.cE[2], 2, k);
        const long long o = zE.s >= 0 ? off_z(d, zE.s, i, j) : 0;
        // E_y is PEC-held where i == 0 or k == 0; E_x where j == 0 or k == 0
        ty = (pi || k == 0) ? T(0) : dbar_c(zE, A1[idk], zE.s >= 0 ? d.apsiE[1][0][o] : T(0));
        tx = (pj || k == 0) ? T(0) : dbar_c(zE, -A0[idk], zE.s >= 0 ? d.apsiE[0][1][o] : T(0));
    };
    T tyz_k, txz_k;
    zterms(z0, id, tyz_k, txz_k);
    for (int k = z0; k < z1; ++k, id += nxy) {
        T tyz_n, txz_n;
        zterms(k + 1, id + nxy, tyz_n, txz_n);
        const bool pk = k == 0;
        const CpmlC<T> zH = cpml_c(d, d.cH[2], 2, k);
        const T b0 = B0[id], b1 = B1[id], b2 = B2[id];
        const T f0 = A0[id], f1 = A1[id], f2 = A2[id];
        const T f2_xp = xe ? A2[id + oxp] : T(0), f1_xp = xe ? A1[id + oxp] : T(0);
        const T f2_yp = ye ? A2[id + oyp] : T(0), f0_yp = ye ? A0[id + oyp] : T(0);
        // E-derivative cotangents: E_e's s = 0 has ybar = +F, s = 1 has ybar = -F; PEC nodes give 0
        // H_x gathers E_y s=0 (z) and E_z s=1 (y); H_y gathers E_z s=0 (x) and E_x s=1 (z);
        // H_z gathers E_x s=0 (y) and E_y s=1 (x)
        // (a +1 neighbour reached by wrapping lies at coordinate 0 of a periodic axis: no PEC)
        const T tzy = (pi || pj) ? T(0)
                                 : dbar_c(yE, -f2, yE.s >= 0 ? d.apsiE[2][1][off_y(d, yE.s, i, k)] : T(0));
        const T tzy_p = (!ye || pi) ? T(0)
                                    : dbar_c(yEp, -f2_yp, yEp.s >= 0 ? d.apsiE[2][1][off_y(d, yEp.s, i, k)] : T(0));
        const T tzx = (pi || pj) ? T(0)
                                 : dbar_c(xE, f2, xE.s >= 0 ? d.apsiE[2][0][off_x(d, xE.s, j, k)] : T(0));
        const T tzx_p = (!xe || pj) ? T(0)
                                    : dbar_c(xEp, f2_xp, xEp.s >= 0 ? d.apsiE[2][0][off_x(d, xEp.s, j, k)] : T(0));
        const T txy = (pk || pj) ? T(0)
                                 : dbar_c(yE, f0, yE.s >= 0 ? d.apsiE[0][0][off_y(d, yE.s, i, k)] : T(0));
        const T txy_p = (!ye || pk) ? T(0)
                                    : dbar_c(yEp, f0_yp, yEp.s >= 0 ? d.apsiE[0][0][off_y(d, yEp.s, i, k)] : T(0));
        const T tyx = (pk || pi) ? T(0)
                                     : dbar_c(xE, -f1, xE.s >= 0 ? d.apsiE[1][1][off_x(d, xE.s, j, k)] : T(0));
        const T tyx_p = (!xe || pk) ? T(0)
                                    : dbar_c(xEp, -f1_xp, xEp.s >= 0 ? d.apsiE[1][1][off_x(d, xEp.s, j, k)] : T(0));
        (void)f1;
        T h0 = b0 + (tyz_k - tyz_n) + (tzy - tzy_p);
        T h1 = b1 + (tzx - tzx_p) + (txz_k - txz_n);
        T h2 = b2 + (txy - txy_p) + (tyx - tyx_p);
        // finish the H-side CPML transpose of step m (k_adj_e(m) has read psibar_H)
        if (yH.s >= 0) {
            T* p = d.apsiH[0][0] + off_y(d, yH.s, i, k);
            *p = yH.b * (*p - S * b0);
            T* q = d.apsiH[2][1] + off_y(d, yH.s, i, k);
            *q = yH.b * (*q + S * b2);
        }
        if (zH.s >= 0) {
            T* p = d.apsiH[0][1] + off_z(d, zH.s, i, j);
            *p = zH.b * (*p + S * b0);
            T* q = d.apsiH[1][0] + off_z(d, zH.s, i, j);
            *q = zH.b * (*q - S * b1);
        }
        if (xH.s >= 0) {
            T* p = d.apsiH[1][1] + off_x(d, xH.s, j, k);
            *p = xH.b * (*p + S * b1);
            T* q = d.apsiH[2][0] + off_x(d, xH.s, j, k);
            *q = xH.b * (*q - S * b2);
        }
        if (mon) {
            h0 += (T)inject_at(d, mons, 3, i, j, k, (long long)(m - 1) * 2 + 1);
            h1 += (T)inject_at(d, mons, 4, i, j, k, (long long)(m - 1) * 2 + 1);
            h2 += (T)inject_at(d, mons, 5, i, j, k, (long long)(m - 1) * 2 + 1);
        }
        B0[id] = h0;
        B1[id] = h1;
        B2[id] = h2;
        tyz_k = tyz_n;
        txz_k = txz_n;
    }
}

template <typename T>
__global__ void __launch_bounds__(kTileX* kTileY, sizeof(T) == 4 ? 3 : 2)
    k_adj_h_gen(const Dom<T>* __restrict__ doms, const Mon* __restrict__ mons, const Tile* __restrict__ tiles, T S,
                int m) {
    const Tile t = tiles[blockIdx.x];
    int i, j;
    tile_coords(t, i, j);
    if (i < 0 || j < 0) return;
    adj_h_column(doms[t.dom], mons, i, j, t.z0, t.z1, t.flags, S, m);
}

// Interior fast paths of the two transposed kernels: tiles that touch no CPML slab, PEC plane,
// domain edge or pole cell.  Without CPML the derivative cotangents reduce to -S Hbar / +S Hbar
// and +F / -F, so k_adj_e_int is the forward E update with Ebar -= S C^- Hbar and
// k_adj_h_int is Hbar += C^+ F.  Loads of a plane are issued before its stores; the z-1
// (z+1) neighbours are carried in registers.  The design-box gradient and the monitor
// injection keep their per-cell checks.
// Interior transposed kernels: bounded so that 4 (FP32) / 3 (FP64) blocks of 256 threads fit an
// SM; left unbounded they take ~140 registers (one block per SM) and starve the memory system.
#ifndef GBFDTD_ADJ_INT_BLOCKS_F32
#define GBFDTD_ADJ_INT_BLOCKS_F32 4
#endif
template <typename T>
constexpr int adj_int_blocks() {
    return sizeof(T) == 4 ? GBFDTD_ADJ_INT_BLOCKS_F32 : 3;
}

template <typename T, bool kAniso>
__global__ void __launch_bounds__(kTileX* kTileY, adj_int_blocks<T>()) k_adj_e_int(const Dom<T>* __restrict__ doms,
                                                              const Mon* __restrict__ mons,
                                                              const Tile* __restrict__ tiles, T S, int m,
                                                              int pending) {
    const Tile t = tiles[blockIdx.x];
    const Dom<T>& d = doms[t.dom];
    const int nx = d.n[0], ny = d.n[1];
    int i, j;
    tile_coords(t, i, j);
    if (i < 0 || j < 0) return;
    const long long nxy = (long long)nx * ny;
    T* Fx = d.A[0];
    T* Fy = d.A[1];
    T* Fz = d.A[2];
    const T* Bx = d.A[3];
    const T* By = d.A[4];
    const T* Bz = d.A[5];
    const T* ie0 = d.ie[0];
    const T* ie1 = d.ie[1];
    const T* ie2 = d.ie[2];
    const bool gcol = d.design && i >= d.glo[0] && i < d.ghi[0] && j >= d.glo[1] && j < d.ghi[1];
    long long id = (long long)t.z0 * nxy + (long long)j * nx + i;
    T bxz = Bx[id - nxy], byz = By[id - nxy];
    for (int k = t.z0; k < t.z1; ++k, id += nxy) {
        const T bx = Bx[id], by = By[id], bz = Bz[id];
        const T bz_ym = Bz[id - nx], bx_ym = Bx[id - nx];
        const T bz_xm = Bz[id - 1], by_xm = By[id - 1];
        const T fx = Fx[id], fy = Fy[id], fz = Fz[id];
        const T iex = ie0[id];
        const T iey = kAniso ? ie1[id] : iex;
        const T iez = kAniso ? ie2[id] : iex;
        // deferred own-cell transpose of step m+1 (non-dispersive: Ebar = F / (S eps^-1))
        T ex = pending ? fx / (S * iex) : fx;
        T ey = pending ? fy / (S * iey) : fy;
        T ez = pending ? fz / (S * iez) : fz;
        // transpose of the H update: Ebar -= S C^- Hbar
        ex += S * ((by - byz) - (bz - bz_ym));
        ey += S * ((bz - bz_xm) - (bx - bxz));
        ez += S * ((bx - bx_ym) - (by - by_xm));
        bxz = bx;
        byz = by;
        if (d.nmon && (t.flags & kTileMonE)) {
            ex += (T)inject_at(d, mons, 0, i, j, k, (long long)m * 2 + 0);
            ey += (T)inject_at(d, mons, 1, i, j, k, (long long)m * 2 + 0);
            ez += (T)inject_at(d, mons, 2, i, j, k, (long long)m * 2 + 0);
        }
        if (gcol && k >= d.glo[2] && k < d.ghi[2]) {
            // d E^{m+1} / d(eps^-1) = S curl(H^{m+1/2}) of the forward state u^m
            const T* Hx = d.F[3];
            const T* Hy = d.F[4];
            const T* Hz = d.F[5];
            const T cx = (Hz[id] - Hz[id - nx]) - (Hy[id] - Hy[id - nxy]);
            const T cy = (Hx[id] - Hx[id - nxy]) - (Hz[id] - Hz[id - 1]);
            const T cz = (Hy[id] - Hy[id - 1]) - (Hx[id] - Hx[id - nx]);
            const long long gi = ((long long)(k - d.glo[2]) * (d.ghi[1] - d.glo[1]) + (j - d.glo[1])) *
                                     (d.ghi[0] - d.glo[0]) + (i - d.glo[0]);
            const long long gn = (long long)(d.ghi[0] - d.glo[0]) * (d.ghi[1] - d.glo[1]) * (d.ghi[2] - d.glo[2]);
            d.grad[gi] += (double)ex * (double)(S * cx);
            d.grad[gn + gi] += (double)ey * (double)(S * cy);
            d.grad[2 * gn + gi] += (double)ez * (double)(S * cz);
        }
        Fx[id] = S * iex * ex;
        Fy[id] = S * iey * ey;
        Fz[id] = S * iez * ez;
    }
}

template <typename T>
__global__ void __launch_bounds__(kTileX* kTileY, adj_int_blocks<T>()) k_adj_h_int(const Dom<T>* __restrict__ doms,
                                                              const Mon* __restrict__ mons,
                                                              const Tile* __restrict__ tiles, T S, int m) {
    const Tile t = tiles[blockIdx.x];
    const Dom<T>& d = doms[t.dom];
    const int nx = d.n[0], ny = d.n[1];
    int i, j;
    tile_coords(t, i, j);
    if (i < 0 || j < 0) return;
    const long long nxy = (long long)nx * ny;
    const T* Fx = d.A[0];
    const T* Fy = d.A[1];
    const T* Fz = d.A[2];
    T* Bx = d.A[3];
    T* By = d.A[4];
    T* Bz = d.A[5];
    long long id = (long long)t.z0 * nxy + (long long)j * nx + i;
    T fxk = Fx[id], fyk = Fy[id];
    for (int k = t.z0; k < t.z1; ++k, id += nxy) {
        const T fxn = Fx[id + nxy], fyn = Fy[id + nxy];
        const T fz = Fz[id];
        const T fz_yp = Fz[id + nx], fz_xp = Fz[id + 1];
        const T fy_xp = Fy[id + 1], fx_yp = Fx[id + nx];
        T bx = Bx[id], by = By[id], bz = Bz[id];
        // transpose of the E update: Hbar += C^+ F
        bx += (fz_yp - fz) - (fyn - fyk);
        by += (fxn - fxk) - (fz_xp - fz);
        bz += (fy_xp - fyk) - (fx_yp - fxk);
        if (d.nmon && m >= 1 && (t.flags & kTileMonH)) {
            bx += (T)inject_at(d, mons, 3, i, j, k, (long long)(m - 1) * 2 + 1);
            by += (T)inject_at(d, mons, 4, i, j, k, (long long)(m - 1) * 2 + 1);
            bz += (T)inject_at(d, mons, 5, i, j, k, (long long)(m - 1) * 2 + 1);
        }
        Bx[id] = bx;
        By[id] = by;
        Bz[id] = bz;
        fxk = fxn;
        fyk = fyn;
    }
}

template <typename T>
__global__ void __launch_bounds__(kTileX* kTileY) k_adj_flush(const Dom<T>* __restrict__ doms,
                                                              const Tile* __restrict__ tiles, T S) {
    const Tile t = tiles[blockIdx.x];
    const Dom<T>& d = doms[t.dom];
    int i, j;
    tile_coords(t, i, j);
    if (i < 0 || j < 0) return;
    for (int k = t.z0; k < t.z1; ++k) {
        const int c[3] = {i, j, k};
        const long long id = cidx(d.n, i, j, k);
        const bool dcell = d.npole > 0 && d.mask[id] && in_ade_box(d, i, j, k);
        for (int a = 0; a < 3; ++a) {
            const int b = (a + 1) % 3, q = (a + 2) % 3;
            if ((c[b] == 0 && !d.per[b]) || (c[q] == 0 && !d.per[q])) continue;   // PEC-held
            d.A[a][id] = e_deferred(d, a, i, j, k, id, dcell, d.A[a][id], S);
        }
    }
}

// Standalone injection of dJ/df(t) into the adjoint fields (used to start a sweep).
template <typename T>
__global__ void k_inject(const Dom<T>* __restrict__ doms, const Mon* __restrict__ mons,
                         const int* __restrict__ entries, int nentries, long long nthreads,
                         const long long* __restrict__ entry_begin, int step, int kind) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= nthreads) return;
    int e = 0;
    while (e + 1 < nentries && entry_begin[e + 1] <= t) ++e;
    const int mi = entries[2 * e], ci = entries[2 * e + 1];
    const Mon& m = mons[mi];
    if (!m.cot) return;
    const long long cell = t - entry_begin[e];
    const int i = m.lo[0] + (int)(cell % m.bx);
    const int j = m.lo[1] + (int)((cell / m.bx) % m.by);
    const int k = m.lo[2] + (int)(cell / ((long long)m.bx * m.by));
    const Dom<T>& d = doms[m.dom];
    const double2* ph = m.phase + ((long long)step * 2 + kind) * m.nf;
    const double2* ct = m.cot + (long long)ci * m.nf * m.ncell + cell;
    double acc = 0.0;
    for (int f = 0; f < m.nf; ++f) {
        const double2 c = ct[(long long)f * m.ncell];
        acc += c.x * ph[f].x + c.y * ph[f].y;
    }
    d.A[m.comps[ci]][cidx(d.n, i, j, k)] += (T)acc;
}

// Injection values of one half-step over a box of cells (see launch_inject_box): the sum over the
// domain's monitors of inject_at, rounded to T once, exactly the value the per-cell kernels add.
template <typename T>
__global__ void k_inject_box(const Dom<T>* __restrict__ dom, const Mon* __restrict__ mons, int3 lo, int3 hi,
                             long long pidx_e, long long pidx_h, T* __restrict__ inj) {
    const long long bx = hi.x - lo.x, by = hi.y - lo.y, vol = bx * by * (hi.z - lo.z);
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= vol) return;
    const int i = lo.x + (int)(t % bx), j = lo.y + (int)((t / bx) % by), k = lo.z + (int)(t / (bx * by));
    for (int c = 0; c < 3; ++c) inj[c * vol + t] = (T)inject_at(*dom, mons, c, i, j, k, pidx_e);
    if (pidx_h >= 0)
        for (int c = 3; c < 6; ++c) inj[c * vol + t] = (T)inject_at(*dom, mons, c, i, j, k, pidx_h);
}

// ---- per-cell transposed kernels -------------------------------------------------------------------
// One thread per cell over a box of blocks of 16 x 16 cells of a plane (the box of the cells with poles or a
// material cotangent, or a whole tensor domain; all other cells run in groups, below), every load of a
// thread independent, the operands by value.  The algebra is that of adj_e_column / adj_h_column: a gathered
// derivative cotangent is Dbar = ybar outside the CPML slabs and ybar / kappa + c (psibar + ybar) in them, decided
// per cell and axis; poles, the material cotangent, pole-coefficient cotangents and monitor injection are compiled
// in only where a domain needs them.
#ifndef GBFDTD_ADJ_CELL_BLOCKS_F32
#define GBFDTD_ADJ_CELL_BLOCKS_F32 8
#endif
template <typename T, bool kHeavy>
constexpr int adj_cell_blocks() {
    return sizeof(T) == 4 ? (kHeavy ? 4 : GBFDTD_ADJ_CELL_BLOCKS_F32) : 3;
}

// Offset of cell (i, j, k) in the slab array of axis q at slab index s, written so that the part
// depending only on the block's plane k (block-uniform) is computed in 64 bits once and the in-plane
// part in 32 bits.
__device__ __forceinline__ int slab_off_c(const int* n, const int* ns, int q, int i, int j, int k, int s) {
    if (q == 0) return k * (n[1] * ns[0]) + (j * ns[0] + s);
    if (q == 1) return k * (ns[1] * n[0]) + (s * n[0] + i);
    return s * (n[0] * n[1]) + (j * n[0] + i);
}

// Dbar of a derivative at node (i, j, k) whose coordinate along axis q is x and slab index sl
// (-1 outside the slabs) and whose ybar is s v: coef is the axis' CPML row [b | c | 1/kappa], psi its memory cotangents.
template <typename T>
__device__ __forceinline__ T dbar_node(const T* coef, int N, const T* psi, const int* n, const int* ns, int q, int i,
                                       int j, int k, int x, int sl, T s, T v) {
    const T yb = mul_t(s, v);
    if (sl < 0) return yb;
    const T ps = psi[slab_off_c(n, ns, q, i, j, k, sl)];
    return fma_t(coef[2 * N + x], yb, mul_t(coef[N + x], ps + yb));
}

// Sum of a component's two gathered cotangents v0, v1 (one per axis): differences of the H cotangents, still to be
// multiplied by S, or (d0, d1) differences of Dbar.  The sum carries the factor S if both are of the first kind, else 1, and
// enters Ebar by one fused multiply-add: no product S v is rounded by itself (rounding them took FP32 transposed fields and
// gradients 1 to 6% further from their FP64 values).
template <typename T>
__device__ __forceinline__ T gathered(T S, bool d0, T v0, bool d1, T v1) {
    return d1 ? fma_t(d0 ? T(1) : S, v0, v1) : fma_t(d0 ? S : T(1), v1, v0);
}

__device__ __forceinline__ bool in_box3(const int* lo, const int* hi, int i, int j, int k) {
    return i >= lo[0] && i < hi[0] && j >= lo[1] && j < hi[1] && k >= lo[2] && k < hi[2];
}

// Offset of cell (i, j, k) inside the box [lo, hi), x fastest.
__device__ __forceinline__ long long box_cell(const int* lo, const int* hi, int i, int j, int k) {
    return ((long long)(k - lo[2]) * (hi[1] - lo[1]) + (j - lo[1])) * (hi[0] - lo[0]) + (i - lo[0]);
}

// 1 / x: a correctly rounded reciprocal in FP32 (a multiply by it replaces the IEEE division of
// the deferred own-cell part), the exact quotient in FP64.
__device__ __forceinline__ float recip_t(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip_t(double x) { return 1.0 / x; }

// Slab index of coordinate x along an axis with CPML depths (lo, hi) over N nodes, or -1; an axis
// without CPML (ns = 0) has none.
__device__ __forceinline__ int slab_or_none(int x, int lo, int hi, int N, int ns) {
    return ns ? slab_of(x, lo, hi, N) : -1;
}

// One E component a of the transposed E step at cell (i, j, k) (offset id of the whole array):
// completes the deferred own-cell transpose of step m+1 (pending), adds the gathered cotangent gs gat (see gathered)
// and the monitor injection, accumulates the material (and pole-coefficient) cotangents, and
// returns the new lagged value S eps^-1 / (1 + eps^-1 G) Ebar.  om: offsets to the -1 neighbours.
// kTen (a tensor domain, Sec. 2.3): Ebar of step m+1 is kept in c.Eb (the pending part only advances
// the psibar_E with F, the curl cotangent the apply kernel left in the E array) and the return value
// is Ebar itself, which the caller stores into c.Eb.
template <typename T, int a, bool kPoles, bool kGrad, bool kMon, int kPG, bool kTen = false>
__device__ __forceinline__ T adj_e_comp(const AdjCellArgs<T>& c, const Dom<T>* __restrict__ doms,
                                        const Mon* __restrict__ mons, int i, int j, int k, long long id, T F, T ie,
                                        T gs, T gat, T S, int m, int pending, bool disp, long long bo,
                                        const int* sl, const long long* om, double* pacc) {
    constexpr int q0 = (a + 1) % 3, q1 = (a + 2) % 3;
    const int x[3] = {i, j, k + c.kz0};   // coefficient rows are indexed by global coordinates
    T eb;
    if (pending) {
        if (kTen) {
            eb = c.Eb[a][id];
        } else if (kPoles && disp) {
            const Dom<T>& d = doms[c.dom];
            eb = (T(1) / ie - d.G) / S * F;
            for (int p = 0; p < d.npole; ++p) {
                T* pp = d.aade + ((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo;
                T* pq = pp + d.bcell;
                const T xp = *pp, xq = *pq;
                eb += d.g0[p] * xp + d.g1[p] * xq;
                *pp = d.M00[p] * xp + d.M10[p] * xq + (T(1) - d.M00[p]) / S * F;
                *pq = d.M01[p] * xp + d.M11[p] * xq - d.M01[p] / S * F;
            }
        } else {
            eb = mul_t(F, recip_t(mul_t(S, ie)));
        }
        // own psibar_E of E_a's two derivatives: s = 0 along q0 (ybar = +F), s = 1 along q1 (-F)
        if (sl[q0] >= 0) {
            T* p = c.apsiE[a][0] + slab_off_c(c.n, c.ns, q0, i, j, k, sl[q0]);
            *p = mul_t(c.cE[q0][x[q0]], *p + F);
        }
        if (sl[q1] >= 0) {
            T* p = c.apsiE[a][1] + slab_off_c(c.n, c.ns, q1, i, j, k, sl[q1]);
            *p = mul_t(c.cE[q1][x[q1]], *p - F);
        }
    } else {
        eb = F;
    }
    eb = fma_t(gs, gat, eb);
    if (kMon && in_box3(c.mlo, c.mhi, i, j, k + c.kz0)) eb += c.inj[a * c.mvol + box_cell(c.mlo, c.mhi, i, j, k + c.kz0)];
    T et = eb, gdisp = T(0);
    if (kPoles && disp) {
        const Dom<T>& d = doms[c.dom];
        for (int p = 0; p < d.npole; ++p) {
            const T* pp = d.aade + ((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo;
            et += d.g0[p] * pp[0] + d.g1[p] * pp[d.bcell];
        }
        gdisp = d.G;
    }
    const bool gcell = kGrad && in_box3(c.glo, c.ghi, i, j, k);
    const bool pcell = kPG != 0 && disp;
    if (gcell || pcell) {
        // d E^{m+1} / d(eps^-1): S curl(H^{m+1/2}) of the forward state u^m (plus the pole terms);
        // the design and pole boxes lie outside the CPML slabs, so the forward update used the
        // plain curl
        const T* Hq = c.F[3 + q1];
        const T* Hb = c.F[3 + q0];
        const T curl = (Hq[id] - Hq[id + om[q0]]) - (Hb[id] - Hb[id + om[q1]]);
        double delta = (double)(S * curl);
        const T e0 = c.F[a][id];
        if (kPoles && disp) {
            const Dom<T>& d = doms[c.dom];
            for (int p = 0; p < d.npole; ++p) {
                const T P = d.ade[((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo];
                const T Q = d.ade[((long long)(a * d.npole + p) * 2 + 1) * d.bcell + bo];
                delta += (double)(P - (d.M00[p] * P + d.M01[p] * Q) - T(2) * d.g0[p] * e0);
            }
        }
        // (1 in a nondispersive cell: no FP64 division there, which on this part costs more than the rest of the cell)
        const bool pol = kPoles && disp;
        const double r = pol ? 1.0 / (1.0 + (double)ie * (double)gdisp) : 1.0;
        if (gcell) {
            const long long gi = ((long long)(k + c.kz0 - c.gzg) * (c.ghi[1] - c.glo[1]) + (j - c.glo[1])) *
                                     (c.ghi[0] - c.glo[0]) + (i - c.glo[0]);
            const double g = (double)et * delta;
            c.grad[a * c.gvol + gi] += pol ? g * r * r : g;
        }
        if (pcell) {
            // pole-coefficient cotangents (the algebra of adj_e_column): with u = xbar_P - rho et,
            //   M00 += u P, M01 += u Q, M10 += xbar_Q P, M11 += xbar_Q Q, g0 += u es, g1 += xbar_Q es
            const Dom<T>& d = doms[c.dom];
            const double rho = (double)ie * r;
            const double es = 2.0 * (double)e0 + rho * delta;
            const double etr = (double)et * rho;
            const int np = kPG == 2 ? 2 : d.npole;
#pragma unroll
            for (int p = 0; p < np; ++p) {
                const long long o0 = ((long long)(a * np + p) * 2 + 0) * d.bcell + bo;
                const long long o1 = o0 + d.bcell;
                const double P = (double)d.ade[o0], Q = (double)d.ade[o1];
                const double xq = (double)d.aade[o1];
                const double u = (double)d.aade[o0] - etr;
                double* pa = pacc + 6 * p;
                pa[0] += u * P;
                pa[1] += u * Q;
                pa[2] += xq * P;
                pa[3] += xq * Q;
                pa[4] += u * es;
                pa[5] += xq * es;
            }
        }
    }
    if (kTen) return et;
    if (kPoles && disp) return S * ie / (T(1) + ie * gdisp) * et;
    return mul_t(mul_t(S, ie), et);
}

// kPG (with kPoles): also sums the pole-coefficient cotangents of the domain (Sec. 3.1: pole parameters
// through the transposed dispersion update): per thread, then one warp sum, a block sum in shared
// memory and one FP64 atomic per block and coefficient into the domain's accumulator.
template <typename T, bool kPoles, bool kGrad, bool kMon, int kPG, bool kTen>
__device__ __forceinline__ void adj_e_cell_body(const AdjCellArgs<T>& c, const Dom<T>* __restrict__ doms,
                                                const Mon* __restrict__ mons, T S, int m, int pending, double* pacc) {
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    // a warp covers 16 x 2 cells (two half-rows of 64 / 128 aligned bytes); the grid covers the box [wlo, whi)
    const int i = c.wlo[0] + blockIdx.x * 16 + (threadIdx.x & 15);
    const int j = c.wlo[1] + blockIdx.y * 16 + threadIdx.y * 2 + (threadIdx.x >> 4);
    const int k = c.wlo[2] + blockIdx.z;
    if (i >= c.whi[0] || j >= c.whi[1]) return;
    const int kg = k + c.kz0;   // global plane (CPML z profile, monitors, plain ranges)
    const long long nxy = (long long)nx * ny;
    const long long pl = (long long)k * nxy;   // first cell of this z-plane (block-uniform)
    const int ij = j * nx + i;                  // offset inside the plane
    // -1 neighbours (wrapping on a periodic axis); in-plane offsets in 32 bits
    const bool hx_ = i > 0 || c.per[0], hy_ = j > 0 || c.per[1], hz_ = k > 0;
    const int ox = i > 0 ? -1 : nx - 1, oy = j > 0 ? -nx : (ny - 1) * nx;
    pdl_wait();
    pdl_trigger();
    const T* Bx = c.A[3] + pl;
    const T* By = c.A[4] + pl;
    const T* Bz = c.A[5] + pl;
    const T bx = Bx[ij], by = By[ij], bz = Bz[ij];
    const T by_zm = hz_ ? (By - nxy)[ij] : T(0), bx_zm = hz_ ? (Bx - nxy)[ij] : T(0);
    const T bz_ym = hy_ ? Bz[ij + oy] : T(0), bx_ym = hy_ ? Bx[ij + oy] : T(0);
    const T bz_xm = hx_ ? Bz[ij + ox] : T(0), by_xm = hx_ ? By[ij + ox] : T(0);
    const T f0 = (c.A[0] + pl)[ij], f1 = (c.A[1] + pl)[ij], f2 = (c.A[2] + pl)[ij];
    const bool aniso = c.ie[1] != c.ie[0] || c.ie[2] != c.ie[0];
    const T ie0 = kTen ? T(1) : (c.ie[0] + pl)[ij];
    const T ie1 = kTen ? T(1) : (aniso ? (c.ie[1] + pl)[ij] : ie0);
    const T ie2 = kTen ? T(1) : (aniso ? (c.ie[2] + pl)[ij] : ie0);
    // where the new E cotangents go: the lagged form into the E array, a tensor domain's Ebar into Eb
    T* const E0 = kTen ? c.Eb[0] : c.A[0];
    T* const E1 = kTen ? c.Eb[1] : c.A[1];
    T* const E2 = kTen ? c.Eb[2] : c.A[2];
    const bool pi = i == 0 && !c.per[0], pj = j == 0 && !c.per[1], pk = k == 0;
    const long long id = pl + ij;
    const long long om[3] = {ox, oy, -nxy};
    bool disp = false;
    long long bo = 0;
    if (kPoles) {
        const Dom<T>& d = doms[c.dom];
        disp = d.npole > 0 && in_ade_box(d, i, j, k) && d.mask[pl + ij];
        if (disp) bo = ade_off(d, i, j, k);
    }
    // a warp (one x row of one plane) whose cells all gather no slab node takes the plain form: the
    // derivative cotangents are S times differences of the H cotangent, and no psibar is touched
    const unsigned am = __activemask();
    const bool plain = (unsigned)(i - c.elo[0]) < (unsigned)(c.ehi[0] - c.elo[0]) &&
                       (unsigned)(j - c.elo[1]) < (unsigned)(c.ehi[1] - c.elo[1]) &&
                       (unsigned)(kg - c.elo[2]) < (unsigned)(c.ehi[2] - c.elo[2]);
    int sl[3] = {-1, -1, -1};
    // the gathered cotangents and their factors (see gathered)
    T g0, g1, g2, s0 = S, s1 = S, s2 = S;
    if (__all_sync(am, plain)) {
        g0 = (by - by_zm) + (bz_ym - bz);
        g1 = (bx_zm - bx) + (bz - bz_xm);
        g2 = (bx - bx_ym) + (by_xm - by);
    } else {
        // slab index of this node along each axis (-1: outside the slabs); the -1 node lies in a slab only where this
        // node is the first one past the low slab
        sl[0] = slab_or_none(i, c.dlo[0], c.dhi[0], nx, c.ns[0]);
        sl[1] = slab_or_none(j, c.dlo[1], c.dhi[1], ny, c.ns[1]);
        sl[2] = slab_or_none(kg, c.dlo[2], c.dhi[2], c.nzg, c.ns[2]);
        // gathered transposes of the H update's derivatives: the q-derivative of H_c has ybar = -S Hbar_c for s = 0 of H_c
        // and +S Hbar_c for s = 1; E_a gathers its two curl terms at this node and at -1: per axis differences of the H
        // cotangents, or of Dbar where a slab node is among the two (dx, dy, dz)
        const bool dz = !(sl[2] < 0 && !(k > 0 && kg == c.dlo[2]));
        const bool dy = !(sl[1] < 0 && !(j > 0 && j == c.dlo[1]));
        const bool dx = !(sl[0] < 0 && !(i > 0 && i == c.dlo[0]));
        T z0 = by - by_zm, z1 = bx_zm - bx;
        // z: H_y (s = 0) into E_x, H_x (s = 1) into E_y
        if (dz) {
            const int szm = k > 0 ? slab_or_none(kg - 1, c.dlo[2], c.dhi[2], c.nzg, c.ns[2]) : -1;
            const T tyz = dbar_node(c.cH[2], c.nzg, c.apsiH[1][0], c.n, c.ns, 2, i, j, k, kg, sl[2], -S, by);
            const T tyz_m = hz_ ? dbar_node(c.cH[2], c.nzg, c.apsiH[1][0], c.n, c.ns, 2, i, j, k - 1, kg - 1, szm, -S, by_zm) : T(0);
            const T txz = dbar_node(c.cH[2], c.nzg, c.apsiH[0][1], c.n, c.ns, 2, i, j, k, kg, sl[2], S, bx);
            const T txz_m = hz_ ? dbar_node(c.cH[2], c.nzg, c.apsiH[0][1], c.n, c.ns, 2, i, j, k - 1, kg - 1, szm, S, bx_zm) : T(0);
            z0 = tyz_m - tyz;
            z1 = txz_m - txz;
        }
        T y0 = bz_ym - bz, y1 = bx - bx_ym;
        // y: H_z (s = 1) into E_x, H_x (s = 0) into E_z
        if (dy) {
            const int sym = j > 0 ? slab_or_none(j - 1, c.dlo[1], c.dhi[1], ny, c.ns[1]) : -1;
            const T tzy = dbar_node(c.cH[1], c.n[1], c.apsiH[2][1], c.n, c.ns, 1, i, j, k, j, sl[1], S, bz);
            const T tzy_m = hy_ ? dbar_node(c.cH[1], c.n[1], c.apsiH[2][1], c.n, c.ns, 1, i, j - 1, k, j - 1, sym, S, bz_ym) : T(0);
            const T txy = dbar_node(c.cH[1], c.n[1], c.apsiH[0][0], c.n, c.ns, 1, i, j, k, j, sl[1], -S, bx);
            const T txy_m = hy_ ? dbar_node(c.cH[1], c.n[1], c.apsiH[0][0], c.n, c.ns, 1, i, j - 1, k, j - 1, sym, -S, bx_ym) : T(0);
            y0 = tzy_m - tzy;
            y1 = txy_m - txy;
        }
        g0 = gathered(S, dz, z0, dy, y0);
        T x0 = bz - bz_xm, x1 = by_xm - by;
        // x: H_z (s = 0) into E_y, H_y (s = 1) into E_z
        if (dx) {
            const int sxm = i > 0 ? slab_or_none(i - 1, c.dlo[0], c.dhi[0], nx, c.ns[0]) : -1;
            const T tzx = dbar_node(c.cH[0], c.n[0], c.apsiH[2][0], c.n, c.ns, 0, i, j, k, i, sl[0], -S, bz);
            const T tzx_m = hx_ ? dbar_node(c.cH[0], c.n[0], c.apsiH[2][0], c.n, c.ns, 0, i - 1, j, k, i - 1, sxm, -S, bz_xm) : T(0);
            const T tyx = dbar_node(c.cH[0], c.n[0], c.apsiH[1][1], c.n, c.ns, 0, i, j, k, i, sl[0], S, by);
            const T tyx_m = hx_ ? dbar_node(c.cH[0], c.n[0], c.apsiH[1][1], c.n, c.ns, 0, i - 1, j, k, i - 1, sxm, S, by_xm) : T(0);
            x0 = tzx_m - tzx;
            x1 = tyx_m - tyx;
        }
        g1 = gathered(S, dz, z1, dx, x0);
        g2 = gathered(S, dy, y1, dx, x1);
        if (dz || dy) s0 = T(1);
        if (dz || dx) s1 = T(1);
        if (dy || dx) s2 = T(1);
    }
    // tangential E on a PEC plane (coordinate 0 of a non-periodic axis other than its own) is held
    if (!(pj || pk))
        (E0 + pl)[ij] = adj_e_comp<T, 0, kPoles, kGrad, kMon, kPG, kTen>(c, doms, mons, i, j, k, id, f0, ie0, s0, g0, S, m,
                                                                      pending, disp, bo, sl, om, pacc);
    if (!(pi || pk))
        (E1 + pl)[ij] = adj_e_comp<T, 1, kPoles, kGrad, kMon, kPG, kTen>(c, doms, mons, i, j, k, id, f1, ie1, s1, g1, S, m,
                                                                      pending, disp, bo, sl, om, pacc);
    if (!(pi || pj))
        (E2 + pl)[ij] = adj_e_comp<T, 2, kPoles, kGrad, kMon, kPG, kTen>(c, doms, mons, i, j, k, id, f2, ie2, s2, g2, S, m,
                                                                      pending, disp, bo, sl, om, pacc);
}

template <typename T, bool kPoles, bool kGrad, bool kMon, int kPG, bool kTen = false>
__global__ void __launch_bounds__(kTileX* kTileY, kPG == 2 ? adj_cell_blocks<T, true>() - 1 : adj_cell_blocks<T, kPoles || kGrad>())
    k_adj_e_cell(const AdjCellArgs<T> c, const Dom<T>* __restrict__ doms, const Mon* __restrict__ mons, T S, int m,
                 int pending) {
    if (!kPG) {
        adj_e_cell_body<T, kPoles, kGrad, kMon, 0, kTen>(c, doms, mons, S, m, pending, nullptr);
        return;
    }
    const Dom<T>& d = doms[c.dom];
    const int np = d.pgc ? d.npole : 0;
    // a block of 16 x 16 cells of one plane that meets no pole-box cell has no pole-coefficient
    // cotangent to add (a block-uniform test): it runs the plain body and skips the reductions
    {
        const int i0 = c.wlo[0] + blockIdx.x * 16, j0 = c.wlo[1] + blockIdx.y * 16, k = c.wlo[2] + blockIdx.z;
        const bool meets = np > 0 && i0 < d.bhi[0] && i0 + 16 > d.blo[0] && j0 < d.bhi[1] && j0 + 16 > d.blo[1] &&
                           k >= d.blo[2] && k < d.bhi[2];
        if (!meets) {
            adj_e_cell_body<T, kPoles, kGrad, kMon, 0, kTen>(c, doms, mons, S, m, pending, nullptr);
            return;
        }
    }
    // every thread of the block reaches the reductions below (the domain, hence np, is the launch's)
    const int tid = threadIdx.y * kTileX + threadIdx.x, lane = tid & 31;
    if (kPG == 2) {
        // two poles: the 12 sums stay in registers, and a warp adds them by halving the slots a lane holds with every
        // exchange (16 FP64 additions a lane instead of 60)
        double v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = 0.0;
        adj_e_cell_body<T, kPoles, kGrad, kMon, 2, false>(c, doms, mons, S, m, pending, v);
#pragma unroll
        for (int w = 8, o = 16; w >= 1; w /= 2, o /= 2) {
            const bool high = lane & o;
#pragma unroll
            for (int q = 0; q < w; ++q) {
                const double send = high ? v[q] : v[q + w], keep = high ? v[q + w] : v[q];
                v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        const int slot = (lane & 16 ? 8 : 0) | (lane & 8 ? 4 : 0) | (lane & 4 ? 2 : 0) | (lane & 2 ? 1 : 0);
        __shared__ double sums[kTileX * kTileY / 32][16];
        if (!(lane & 1)) sums[tid >> 5][slot] = v[0];
        __syncthreads();
        if (tid >= 12) return;
        double t = 0.0;
        for (int w = 0; w < kTileX * kTileY / 32; ++w) t += sums[w][tid];
        if (t != 0.0) atomicAdd(d.pgc + tid, t);
        return;
    }
    double acc[kMaxPole * 6];
    for (int q = 0; q < np * 6; ++q) acc[q] = 0.0;
    adj_e_cell_body<T, kPoles, kGrad, kMon, 1, false>(c, doms, mons, S, m, pending, acc);
    __shared__ double red[kTileX * kTileY / 32];
    for (int q = 0; q < np * 6; ++q) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < kTileX * kTileY / 32; ++w) t += red[w];
            if (t != 0.0) atomicAdd(d.pgc + q, t);
        }
        __syncthreads();
    }
}

// ---- transposed updates by groups of cells ------------------------------------------------------------
// The cells that need no pole, material-cotangent or tensor work (all of them but a box, see launch_adj_e_cell), kV
// consecutive cells of a row per thread like the forward updates.  What bounds the scalar form is instruction
// issue.  A plane is cut into three regions of whole blocks, so that the long groups run without any slab code
// and the slab code with whole warps: (0) groups whose gathers meet no slab node, in the columns, rows and planes
// where none does; (1) the other columns; (2) the remaining rows of the first columns (every row of a plane in a z
// slab).  Regions 1 and 2 run kG cells per thread through the general gather, decided per cell and axis.  Every
// form computes the same sums in the same order with spelled-out roundings (see gathered), so a cell's bits do not
// depend on the region, the group length or the kernel.
constexpr int kAdjLong = 4, kAdjShort = 2;   // cells per thread of region 0 and of the others, where they fit

// Blocks per SM, as threads per SM: 64 registers hold a group of four and the slab work of one axis at a time (FP32,
// 128^3 with 10-cell CPML: E 27.7 -> 15.9, H 23.3 -> 14.7 us; 256^3 with 12: 171 -> 129, 149 -> 126; without CPML 128^3
// 15.4 -> 9.9, 12.5 -> 10.2); one cell per thread (odd rows) wants every warp it can get (243 x 251 x 229: 2048 threads
// 129 + 122 us; 1536 were 9% slower; the scalar kernels took 159 + 138).  FP64 is bound by its pipe.
template <typename T, int kV>
constexpr int adj_group_blocks() {
    return (sizeof(T) == 4 ? (kV == 1 ? 2048 : 1024) : 1024) / kCellThreads;
}

struct AdjAt {
    int i, j;
    bool left, right, live;
};

// Thread of block `block` of region r -> its group of v cells (left / right / live as in the forward group_at).
template <typename T, int kV>
__device__ __forceinline__ AdjAt adj_at(const AdjCellArgs<T>& c, int r, unsigned block, bool zplain) {
    const GroupRows& R = c.rows[r];
    const int inner = c.gy1 - c.gy0;   // rows of region 0
    const unsigned nrow = r == 0 ? inner : r == 1 || !zplain ? c.n[1] : c.n[1] - inner;
    const unsigned n = R.gp * nrow;
    unsigned t = block * kCellThreads + threadIdx.x;
    AdjAt g;
    g.live = t < n;
    if (!g.live) t = n - 1;
    const unsigned row = group_row(R, t);
    const int col = (int)(t - row * R.gp), lane = threadIdx.x & 31, x = col * kV;
    g.j = r == 0 ? c.gy0 + (int)row : r == 2 && zplain && (int)row >= c.gy0 ? (int)row + inner : (int)row;
    g.i = r == 1 ? (x < c.gx ? x : x + c.gxn) : c.gx + x;
    g.left = lane != 0 && col != 0 && !(r == 1 && x == c.gx);
    g.right = lane != 31 && col + 1 != (int)R.gp && !(r == 1 && x + kV == c.gx);
    return g;
}

// The slab data of a group along z or y, loaded at once: the two gathered memory cotangents at this node (a, bb) and at
// its neighbour (an, bn), the two own memories (o0, o1) and the coefficients.  (Loading the three axes' data ahead,
// beside the fields, as the forward updates do, took registers from a whole block per SM and was slower: 25.2
// against 22.3 us for E at 128^3.)  Slab indices are -1 outside.
template <typename T, int kV>
struct AdjAxis {
    int s, sn;            // slab index of this node, of the neighbour
    unsigned o, on;       // offsets in the memories
    T c, k, cn, kn, b;    // c, 1 / kappa here and at the neighbour (the gathered side's row), b of the own memories
    Group<T, kV> a, bb, an, bn, o0, o1;
};

// node / nb: coordinates of this node and the neighbour along the axis (nb < 0: none); go: the gathered row [b | c | 1 /
// kappa] of N nodes, ow: the own memories' row.
template <typename T, int kV>
__device__ __forceinline__ void load_axis(AdjAxis<T, kV>& m, int s, int sn, unsigned o, unsigned on, const T* go,
                                          const T* ow, int N, int node, int nb, const T* pa, const T* pb, const T* p0,
                                          const T* p1, bool own) {
    m.s = s;
    m.sn = sn;
    m.o = o;
    m.on = on;
    if (s >= 0) {
        m.a = ld_group<T, kV>(pa + o);
        m.bb = ld_group<T, kV>(pb + o);
        m.c = go[N + node];
        m.k = go[2 * N + node];
        if (own) {
            m.o0 = ld_group<T, kV>(p0 + o);
            m.o1 = ld_group<T, kV>(p1 + o);
            m.b = ow[node];
        }
    }
    if (sn >= 0) {
        m.an = ld_group<T, kV>(pa + on);
        m.bn = ld_group<T, kV>(pb + on);
        m.cn = go[N + nb];
        m.kn = go[2 * N + nb];
    }
}
// Dbar of a derivative whose ybar is yb at a node with coefficients c, 1 / kappa and memory cotangent ps.
template <typename T, int kV>
__device__ __forceinline__ Group<T, kV> dbar_of(T cc, T kk, const Group<T, kV>& ps, const Group<T, kV>& yb) {
    Group<T, kV> d;
#pragma unroll
    for (int q = 0; q < kV; ++q) d[q] = fma_t(kk, yb[q], mul_t(cc, ps[q] + yb[q]));
    return d;
}
template <typename T, int kV>
__device__ __forceinline__ Group<T, kV> scaled(T s, const Group<T, kV>& g) {
    Group<T, kV> d;
#pragma unroll
    for (int q = 0; q < kV; ++q) d[q] = mul_t(s, g[q]);
    return d;
}
template <typename T, int kV>
__device__ __forceinline__ Group<T, kV> minus(const Group<T, kV>& a, const Group<T, kV>& b) {
    Group<T, kV> d;
#pragma unroll
    for (int q = 0; q < kV; ++q) d[q] = a[q] - b[q];
    return d;
}
template <typename T, int kV>
__device__ __forceinline__ Group<T, kV> plus(const Group<T, kV>& a, const Group<T, kV>& b) {
    Group<T, kV> d;
#pragma unroll
    for (int q = 0; q < kV; ++q) d[q] = a[q] + b[q];
    return d;
}

// p <- b (p + s v) of the cells not held (bits of hold), stored at psi.
template <typename T, int kV>
__device__ __forceinline__ void psi_group(T* psi, Group<T, kV> p, T b, T s, const Group<T, kV>& v, unsigned hold) {
#pragma unroll
    for (int q = 0; q < kV; ++q)
        if (!(hold >> q & 1)) p[q] = mul_t(b, fma_t(s, v[q], p[q]));
    st_group(psi, p);
}

// The x-slab data of a group's cells (region 1): slab indices of each node and its neighbour, the gathered memory
// cotangents there and the own memories.
template <typename T, int kV>
struct AdjEdge {
    int s[kV], sn[kV];
    Group<T, kV> a, b, an, bn, o0, o1;
};
// step: -1 (the E side gathers the -1 neighbour) or +1; row: offset of slab index 0 of this row.
template <typename T, int kV>
__device__ __forceinline__ void load_edge(const AdjCellArgs<T>& c, AdjEdge<T, kV>& m, int i, int step, unsigned row,
                                          const T* pa, const T* pb, const T* p0, const T* p1, bool own) {
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        const int x = i + q, y = x + step, nx = c.n[0];
        m.s[q] = c.ns[0] ? slab_of(x, c.dlo[0], c.dhi[0], nx) : -1;
        m.sn[q] = c.ns[0] && y >= 0 && y < nx ? slab_of(y, c.dlo[0], c.dhi[0], nx) : -1;
        if (m.s[q] >= 0) {
            m.a[q] = pa[row + m.s[q]];
            m.b[q] = pb[row + m.s[q]];
            if (own) {
                m.o0[q] = p0[row + m.s[q]];
                m.o1[q] = p1[row + m.s[q]];
            }
        }
        if (m.sn[q] >= 0) {
            m.an[q] = pa[row + m.sn[q]];
            m.bn[q] = pb[row + m.sn[q]];
        }
    }
}
template <typename T>
__device__ __forceinline__ T dbar_x(const T* coef, int nx, int x, int sl, T ps, T s, T v) {
    const T yb = mul_t(s, v);
    return sl < 0 ? yb : fma_t(coef[2 * nx + x], yb, mul_t(coef[nx + x], ps + yb));
}

// Transposed E step of a group: gathers the derivative cotangents of the H update, completes the deferred own-cell
// part of step m + 1 (pending), adds the monitor injection and leaves the lagged cotangent S eps^-1 Ebar.
template <typename T, int kV, bool kGeneral, bool kX, bool kAniso, bool kMon>
__device__ __forceinline__ void adj_e_group(const AdjCellArgs<T>& c, T S, int pending, const AdjAt& at, int k) {
    using G = Group<T, kV>;
    const int nx = c.n[0], ny = c.n[1], i = at.i, j = at.j, kg = k + c.kz0;
    const long long nxy = (long long)nx * ny;
    const long long id = (long long)k * nxy + (j * nx + i);
    const T* Bx = c.A[3] + id;
    const T* By = c.A[4] + id;
    const T* Bz = c.A[5] + id;
    const G bx = ld_group<T, kV>(Bx), by = ld_group<T, kV>(By), bz = ld_group<T, kV>(Bz);
    G bx_zm{}, by_zm{}, bx_ym{}, bz_ym{}, by_xm{}, bz_xm{};
    if (k > 0) {
        bx_zm = ld_group<T, kV>(Bx - nxy);
        by_zm = ld_group<T, kV>(By - nxy);
    }
    const bool hy_ = j > 0 || c.per[1], hx_ = i > 0 || c.per[0];   // the -1 neighbours exist (or wrap)
    if (hy_) {
        const long long o = j > 0 ? -(long long)nx : nxy - nx;
        bx_ym = ld_group<T, kV>(Bx + o);
        bz_ym = ld_group<T, kV>(Bz + o);
    }
    T bzl = T(0), byl = T(0);
    if (i == 0 ? (bool)c.per[0] : !at.left) {
        const int o = i == 0 ? nx - 1 : -1;
        bzl = Bz[o];
        byl = By[o];
    }
    G f0 = ld_group<T, kV>(c.A[0] + id), f1 = ld_group<T, kV>(c.A[1] + id), f2 = ld_group<T, kV>(c.A[2] + id);
    const G ie0 = ld_group<T, kV>(c.ie[0] + id);
    const G ie1 = kAniso ? ld_group<T, kV>(c.ie[1] + id) : ie0, ie2 = kAniso ? ld_group<T, kV>(c.ie[2] + id) : ie0;
    const T zl = __shfl_up_sync(0xffffffffu, bz[kV - 1], 1), yl = __shfl_up_sync(0xffffffffu, by[kV - 1], 1);
    if (!at.live) return;
    // the heavy kernel's box (a group lies in it whole or not at all)
    if (i >= c.wlo[0] && i < c.whi[0] && j >= c.wlo[1] && j < c.whi[1] && k >= c.wlo[2] && k < c.whi[2]) return;
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        bz_xm[q] = q ? bz[q ? q - 1 : 0] : at.left && i > 0 ? zl : bzl;
        by_xm[q] = q ? by[q ? q - 1 : 0] : at.left && i > 0 ? yl : byl;
    }
    constexpr unsigned all = (1u << kV) - 1;
    const bool pj = j == 0 && !c.per[1], pk = k == 0;
    const unsigned pi = i == 0 && !c.per[0] ? 1u : 0u;
    const unsigned hold0 = pj || pk ? all : 0u, hold1 = pk ? all : pi, hold2 = pj ? all : pi;   // PEC-held components
    // per axis the differences of the H cotangents, or of the gathered Dbar where a slab node is among the two (see gathered);
    // there (pending) also the own psibar_E of step m + 1: s = 0 takes + F, s = 1 - F.  A component's term of the later axis that
    // is a Dbar joins the earlier one's at once and leaves zero.
    bool dz = false, dy = false;
    unsigned dx = 0;   // cells (bits)
    G z0 = minus(by, by_zm), z1 = minus(bx_zm, bx);
    if (kGeneral) {
        const int sz = c.ns[2] ? slab_of(kg, c.dlo[2], c.dhi[2], c.nzg) : -1;
        const int szm = c.ns[2] && k > 0 ? slab_of(kg - 1, c.dlo[2], c.dhi[2], c.nzg) : -1;
        if (sz >= 0 || szm >= 0) {
            AdjAxis<T, kV> m;
            load_axis(m, sz, szm, ((unsigned)sz * ny + j) * nx + i, ((unsigned)szm * ny + j) * nx + i, c.cH[2], c.cE[2],
                      c.nzg, kg, kg - 1, c.apsiH[1][0], c.apsiH[0][1], c.apsiE[0][1], c.apsiE[1][0], pending);
            G p = scaled(-S, by), pm = scaled(-S, by_zm), r = scaled(S, bx), rm = scaled(S, bx_zm);
            if (sz >= 0) {
                p = dbar_of(m.c, m.k, m.a, p);
                r = dbar_of(m.c, m.k, m.bb, r);
                if (pending) {
                    psi_group(c.apsiE[0][1] + m.o, m.o0, m.b, T(-1), f0, hold0);
                    psi_group(c.apsiE[1][0] + m.o, m.o1, m.b, T(1), f1, hold1);
                }
            }
            if (szm >= 0) {
                pm = dbar_of(m.cn, m.kn, m.an, pm);
                rm = dbar_of(m.cn, m.kn, m.bn, rm);
            }
            z0 = minus(k > 0 ? pm : G{}, p);
            z1 = minus(k > 0 ? rm : G{}, r);
            dz = true;
        }
    }
    G y0 = minus(bz_ym, bz), y1 = minus(bx, bx_ym);
    if (kGeneral) {
        const int sy = c.ns[1] ? slab_of(j, c.dlo[1], c.dhi[1], ny) : -1;
        const int sym = c.ns[1] && j > 0 ? slab_of(j - 1, c.dlo[1], c.dhi[1], ny) : -1;
        if (sy >= 0 || sym >= 0) {
            AdjAxis<T, kV> m;
            load_axis(m, sy, sym, (unsigned)(k * c.ns[1] + sy) * nx + i, (unsigned)(k * c.ns[1] + sym) * nx + i, c.cH[1],
                      c.cE[1], ny, j, j - 1, c.apsiH[2][1], c.apsiH[0][0], c.apsiE[0][0], c.apsiE[2][1], pending);
            G p = scaled(S, bz), pm = scaled(S, bz_ym), r = scaled(-S, bx), rm = scaled(-S, bx_ym);
            if (sy >= 0) {
                p = dbar_of(m.c, m.k, m.a, p);
                r = dbar_of(m.c, m.k, m.bb, r);
                if (pending) {
                    psi_group(c.apsiE[0][0] + m.o, m.o0, m.b, T(1), f0, hold0);
                    psi_group(c.apsiE[2][1] + m.o, m.o1, m.b, T(-1), f2, hold2);
                }
            }
            if (sym >= 0) {
                pm = dbar_of(m.cn, m.kn, m.an, pm);
                rm = dbar_of(m.cn, m.kn, m.bn, rm);
            }
            y0 = minus(hy_ ? pm : G{}, p);
            y1 = minus(hy_ ? rm : G{}, r);
            dy = true;
#pragma unroll
            for (int q = 0; q < kV; ++q) z0[q] = gathered(S, dz, z0[q], true, y0[q]);
            y0 = G{};
        }
    }
    G x0 = minus(bz, bz_xm), x1 = minus(by_xm, by);
    if (kX) {
        AdjEdge<T, kV> m;
        const unsigned row = (unsigned)(k * ny + j) * (unsigned)c.ns[0];
        load_edge(c, m, i, -1, row, c.apsiH[2][0], c.apsiH[1][1], c.apsiE[1][1], c.apsiE[2][0], pending);
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            if (m.s[q] < 0 && m.sn[q] < 0) continue;
            const int x = i + q;
            const bool ex = x > 0 || hx_;
            x0[q] = (ex ? dbar_x(c.cH[0], nx, x - 1, m.sn[q], m.an[q], -S, bz_xm[q]) : T(0)) -
                    dbar_x(c.cH[0], nx, x, m.s[q], m.a[q], -S, bz[q]);
            x1[q] = (ex ? dbar_x(c.cH[0], nx, x - 1, m.sn[q], m.bn[q], S, by_xm[q]) : T(0)) -
                    dbar_x(c.cH[0], nx, x, m.s[q], m.b[q], S, by[q]);
            dx |= 1u << q;
            z1[q] = gathered(S, dz, z1[q], true, x0[q]);
            y1[q] = gathered(S, dy, y1[q], true, x1[q]);
            x0[q] = x1[q] = T(0);
            if (!pending || m.s[q] < 0) continue;
            const T b = c.cE[0][x];
            if (!(hold1 >> q & 1)) c.apsiE[1][1][row + m.s[q]] = mul_t(b, m.o0[q] - f1[q]);
            if (!(hold2 >> q & 1)) c.apsiE[2][0][row + m.s[q]] = mul_t(b, m.o1[q] + f2[q]);
        }
    }
    const bool inj = kMon && kg >= c.mlo[2] && kg < c.mhi[2] && j >= c.mlo[1] && j < c.mhi[1];
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        const T s0 = mul_t(S, ie0[q]), s1 = kAniso ? mul_t(S, ie1[q]) : s0, s2 = kAniso ? mul_t(S, ie2[q]) : s0;
        T e0 = f0[q], e1 = f1[q], e2 = f2[q];
        if (pending) {
            const T r0 = recip_t(s0), r1 = kAniso ? recip_t(s1) : r0, r2 = kAniso ? recip_t(s2) : r0;
            e0 = mul_t(e0, r0);
            e1 = mul_t(e1, r1);
            e2 = mul_t(e2, r2);
        }
        const bool dxq = kX && (dx >> q & 1);
        e0 = fma_t(dz || dy ? T(1) : S, gathered(S, dz, z0[q], false, y0[q]), e0);
        e1 = fma_t(dz || dxq ? T(1) : S, gathered(S, dz, z1[q], false, x0[q]), e1);
        e2 = fma_t(dy || dxq ? T(1) : S, gathered(S, dy, y1[q], false, x1[q]), e2);
        if (inj && i + q >= c.mlo[0] && i + q < c.mhi[0]) {
            const long long bo = box_cell(c.mlo, c.mhi, i + q, j, kg);
            e0 = e0 + c.inj[bo];
            e1 = e1 + c.inj[c.mvol + bo];
            e2 = e2 + c.inj[2 * c.mvol + bo];
        }
        if (!(hold0 >> q & 1)) f0[q] = mul_t(s0, e0);
        if (!(hold1 >> q & 1)) f1[q] = mul_t(s1, e1);
        if (!(hold2 >> q & 1)) f2[q] = mul_t(s2, e2);
    }
    st_group(c.A[0] + id, f0);
    st_group(c.A[1] + id, f1);
    st_group(c.A[2] + id, f2);
}

// Transposed H step of a group: gathers the derivative cotangents of the E update (whose lagged cotangent the E-side
// launch left in the E array), advances the H memories and adds the monitor injection.
template <typename T, int kV, bool kGeneral, bool kX, bool kMon>
__device__ __forceinline__ void adj_h_group(const AdjCellArgs<T>& c, T S, int m, const AdjAt& at, int k) {
    using G = Group<T, kV>;
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2], i = at.i, j = at.j, kg = k + c.kz0;
    const long long nxy = (long long)nx * ny;
    const long long id = (long long)k * nxy + (j * nx + i);
    const T* Fx = c.A[0] + id;
    const T* Fy = c.A[1] + id;
    const T* Fz = c.A[2] + id;
    const G fx = ld_group<T, kV>(Fx), fy = ld_group<T, kV>(Fy), fz = ld_group<T, kV>(Fz);
    const bool ze = k + 1 < nz, ye = j + 1 < ny || c.per[1];
    const bool last = i + kV >= nx, xe = !last || c.per[0];   // the +1 neighbours exist (or wrap); x: of the last cell
    G fx_zp{}, fy_zp{}, fx_yp{}, fz_yp{}, fy_xp{}, fz_xp{};
    if (ze) {
        fx_zp = ld_group<T, kV>(Fx + nxy);
        fy_zp = ld_group<T, kV>(Fy + nxy);
    }
    if (ye) {
        const long long o = j + 1 < ny ? (long long)nx : nx - nxy;
        fx_yp = ld_group<T, kV>(Fx + o);
        fz_yp = ld_group<T, kV>(Fz + o);
    }
    T fzr = T(0), fyr = T(0);
    if (last ? (bool)c.per[0] : !at.right) {
        const int o = last ? kV - nx : kV;
        fzr = Fz[o];
        fyr = Fy[o];
    }
    const G b0 = ld_group<T, kV>(c.A[3] + id), b1 = ld_group<T, kV>(c.A[4] + id), b2 = ld_group<T, kV>(c.A[5] + id);
    const T zr = __shfl_down_sync(0xffffffffu, fz[0], 1), yr = __shfl_down_sync(0xffffffffu, fy[0], 1);
    if (!at.live) return;
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        constexpr int e = kV - 1;
        fz_xp[q] = q < e ? fz[q < e ? q + 1 : 0] : at.right && !last ? zr : fzr;
        fy_xp[q] = q < e ? fy[q < e ? q + 1 : 0] : at.right && !last ? yr : fyr;
    }
    // differences along each axis: z into H_x, H_y; y into H_x, H_z; x into H_y, H_z
    G z0 = minus(fy, fy_zp), z1 = minus(fx_zp, fx);
    G y0 = minus(fz_yp, fz), y2 = minus(fx, fx_yp);
    G x1 = minus(fz, fz_xp), x2 = minus(fy_xp, fy);
    if (kGeneral) {
        const bool pj = j == 0 && !c.per[1], pk = k == 0;
        const bool px = i == 0 && !c.per[0];   // of the first cell
        auto zero_if = [&](G g, bool every, bool first) {   // PEC-held E nodes carry no cotangent
#pragma unroll
            for (int q = 0; q < kV; ++q)
                if (every || (first && q == 0)) g[q] = T(0);
            return g;
        };
        // axis by axis: the gathered Dbar, then the H-side memories of step m (the E-side launch has read them)
        {
            G p = fy, pn = fy_zp, r = scaled(T(-1), fx), rn = scaled(T(-1), fx_zp);   // ybar
            const int sz = c.ns[2] ? slab_of(kg, c.dlo[2], c.dhi[2], c.nzg) : -1;
            const int szp = c.ns[2] && ze ? slab_of(kg + 1, c.dlo[2], c.dhi[2], c.nzg) : -1;
            if (sz >= 0 || szp >= 0) {
                AdjAxis<T, kV> m;
                load_axis(m, sz, szp, ((unsigned)sz * ny + j) * nx + i, ((unsigned)szp * ny + j) * nx + i, c.cE[2],
                          c.cH[2], c.nzg, kg, kg + 1, c.apsiE[1][0], c.apsiE[0][1], c.apsiH[0][1], c.apsiH[1][0], true);
                if (sz >= 0) {
                    p = dbar_of(m.c, m.k, m.a, p);
                    r = dbar_of(m.c, m.k, m.bb, r);
                    psi_group(c.apsiH[0][1] + m.o, m.o0, m.b, S, b0, 0u);
                    psi_group(c.apsiH[1][0] + m.o, m.o1, m.b, -S, b1, 0u);
                }
                if (szp >= 0) {
                    pn = dbar_of(m.cn, m.kn, m.an, pn);
                    rn = dbar_of(m.cn, m.kn, m.bn, rn);
                }
            }
            z0 = minus(zero_if(p, pk, px), zero_if(pn, !ze, px));
            z1 = minus(zero_if(r, pj || pk, false), zero_if(rn, !ze || pj, false));
        }
        {
            G p = scaled(T(-1), fz), pn = scaled(T(-1), fz_yp), r = fx, rn = fx_yp;
            const int sy = c.ns[1] ? slab_of(j, c.dlo[1], c.dhi[1], ny) : -1;
            const int syp = c.ns[1] && j + 1 < ny ? slab_of(j + 1, c.dlo[1], c.dhi[1], ny) : -1;
            if (sy >= 0 || syp >= 0) {
                AdjAxis<T, kV> m;
                load_axis(m, sy, syp, (unsigned)(k * c.ns[1] + sy) * nx + i, (unsigned)(k * c.ns[1] + syp) * nx + i,
                          c.cE[1], c.cH[1], ny, j, j + 1, c.apsiE[2][1], c.apsiE[0][0], c.apsiH[0][0], c.apsiH[2][1],
                          true);
                if (sy >= 0) {
                    p = dbar_of(m.c, m.k, m.a, p);
                    r = dbar_of(m.c, m.k, m.bb, r);
                    psi_group(c.apsiH[0][0] + m.o, m.o0, m.b, -S, b0, 0u);
                    psi_group(c.apsiH[2][1] + m.o, m.o1, m.b, S, b2, 0u);
                }
                if (syp >= 0) {
                    pn = dbar_of(m.cn, m.kn, m.an, pn);
                    rn = dbar_of(m.cn, m.kn, m.bn, rn);
                }
            }
            y0 = minus(zero_if(p, pj, px), zero_if(pn, !ye, px));
            y2 = minus(zero_if(r, pk || pj, false), zero_if(rn, !ye || pk, false));
        }
        AdjEdge<T, kV> m;
        const unsigned row = (unsigned)(k * ny + j) * (unsigned)c.ns[0];
        if (kX) load_edge(c, m, i, 1, row, c.apsiE[2][0], c.apsiE[1][1], c.apsiH[1][1], c.apsiH[2][0], true);
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const int x = i + q;
            const bool first = px && q == 0, has = q < kV - 1 || xe;
            const int sx = kX ? m.s[q] : -1, sxp = kX ? m.sn[q] : -1;
            x1[q] = (first || pj ? T(0) : dbar_x(c.cE[0], nx, x, sx, kX ? m.a[q] : T(0), T(1), fz[q])) -
                    (!has || pj ? T(0) : dbar_x(c.cE[0], nx, x + 1, sxp, kX ? m.an[q] : T(0), T(1), fz_xp[q]));
            x2[q] = (pk || first ? T(0) : dbar_x(c.cE[0], nx, x, sx, kX ? m.b[q] : T(0), T(-1), fy[q])) -
                    (!has || pk ? T(0) : dbar_x(c.cE[0], nx, x + 1, sxp, kX ? m.bn[q] : T(0), T(-1), fy_xp[q]));
            if (sx < 0) continue;
            const T b = c.cH[0][x];
            c.apsiH[1][1][row + (unsigned)sx] = mul_t(b, fma_t(S, b1[q], m.o0[q]));
            c.apsiH[2][0][row + (unsigned)sx] = mul_t(b, fma_t(-S, b2[q], m.o1[q]));
        }
    }
    G h0 = plus(plus(b0, z0), y0), h1 = plus(plus(b1, z1), x1), h2 = plus(plus(b2, y2), x2);
    if (kMon && m >= 1 && kg >= c.mlo[2] && kg < c.mhi[2] && j >= c.mlo[1] && j < c.mhi[1]) {
#pragma unroll
        for (int q = 0; q < kV; ++q)
            if (i + q >= c.mlo[0] && i + q < c.mhi[0]) {
                const long long bo = box_cell(c.mlo, c.mhi, i + q, j, kg);
                h0[q] += c.inj[bo];
                h1[q] += c.inj[c.mvol + bo];
                h2[q] += c.inj[2 * c.mvol + bo];
            }
    }
    st_group(c.A[3] + id, h0);
    st_group(c.A[4] + id, h1);
    st_group(c.A[5] + id, h2);
}

// Region and block of this thread block in plane k; false where the plane has fewer blocks.  hside: plane 0 (held by the
// wall, or a window's cut edge) is no plain plane.
template <typename T>
__device__ __forceinline__ bool adj_region(const AdjCellArgs<T>& c, int k, bool hside, unsigned b, int& r, unsigned& block,
                                           bool& zplain) {
    const int kg = k + c.kz0;
    zplain = kg >= c.gz0 && kg < c.gz1 && !(hside && k == 0);
    const unsigned n0 = zplain ? c.rows[0].nb : 0, n2 = zplain ? c.rows[2].nb : c.nball;
    r = b < n0 ? 0 : b < n0 + c.rows[1].nb ? 1 : 2;
    block = r == 0 ? b : r == 1 ? b - n0 : b - n0 - c.rows[1].nb;
    return r < 2 || block < n2;
}

template <typename T, int kV, int kG, bool kAniso, bool kMon>
__global__ void __launch_bounds__(kCellThreads, adj_group_blocks<T, kV>())
    k_adj_e_group(const __grid_constant__ AdjCellArgs<T> c, T S, int pending) {
    const int k = blockIdx.y;
    int r;
    unsigned block;
    bool zplain;
    const bool any = adj_region(c, k, false, blockIdx.x, r, block, zplain);
    pdl_wait();
    pdl_trigger();
    if (!any) return;
    if (r == 0)
        adj_e_group<T, kV, false, false, kAniso, kMon>(c, S, pending, adj_at<T, kV>(c, 0, block, zplain), k);
    else if (r == 1)
        adj_e_group<T, kG, true, true, kAniso, kMon>(c, S, pending, adj_at<T, kG>(c, 1, block, zplain), k);
    else
        adj_e_group<T, kG, true, false, kAniso, kMon>(c, S, pending, adj_at<T, kG>(c, 2, block, zplain), k);
}

template <typename T, int kV, int kG, bool kMon>
__global__ void __launch_bounds__(kCellThreads, adj_group_blocks<T, kV>())
    k_adj_h_group(const __grid_constant__ AdjCellArgs<T> c, T S, int m) {
    const int k = (int)(gridDim.y - 1 - blockIdx.y);   // last plane first: what the E side has just touched is in L2
    int r;
    unsigned block;
    bool zplain;
    const bool any = adj_region(c, k, true, blockIdx.x, r, block, zplain);
    pdl_wait();
    pdl_trigger();
    if (!any) return;
    if (r == 0)
        adj_h_group<T, kV, false, false, kMon>(c, S, m, adj_at<T, kV>(c, 0, block, zplain), k);
    else if (r == 1)
        adj_h_group<T, kG, true, true, kMon>(c, S, m, adj_at<T, kG>(c, 1, block, zplain), k);
    else
        adj_h_group<T, kG, true, false, kMon>(c, S, m, adj_at<T, kG>(c, 2, block, zplain), k);
}

// Completes a pending transposed step cell by cell (the algebra of e_deferred): for every E
// component not held by a PEC plane, Ebar = F / (S eps^-1) (or the pole form in dispersive cells,
// which also advances the pole cotangents) and the own psibar_E of its two derivatives.
template <typename T, bool kPoles, bool kTen = false>
__global__ void __launch_bounds__(kTileX* kTileY) k_adj_flush_cell(const AdjCellArgs<T> c,
                                                                   const Dom<T>* __restrict__ doms, T S) {
    const int nx = c.n[0], ny = c.n[1];
    const int i = blockIdx.x * kTileX + threadIdx.x, j = blockIdx.y * kTileY + threadIdx.y, k = blockIdx.z;
    if (i >= nx || j >= ny) return;
    const int kg = k + c.kz0;
    const long long id = ((long long)k * ny + j) * nx + i;
    const int sl[3] = {slab_or_none(i, c.dlo[0], c.dhi[0], nx, c.ns[0]), slab_or_none(j, c.dlo[1], c.dhi[1], ny, c.ns[1]),
                       slab_or_none(kg, c.dlo[2], c.dhi[2], c.nzg, c.ns[2])};
    const int x[3] = {i, j, kg};
    bool disp = false;
    long long bo = 0;
    if (kPoles) {
        const Dom<T>& d = doms[c.dom];
        disp = d.npole > 0 && in_ade_box(d, i, j, k) && d.mask[id];
        if (disp) bo = ade_off(d, i, j, k);
    }
    const bool pi = i == 0 && !c.per[0], pj = j == 0 && !c.per[1], pk = k == 0;
    const bool pec[3] = {pj || pk, pi || pk, pi || pj};
    for (int a = 0; a < 3; ++a) {
        if (pec[a]) continue;
        const T ie = kTen ? T(1) : c.ie[a][id];
        const T F = c.A[a][id];
        T eb;
        if (kTen) {
            eb = c.Eb[a][id];
        } else if (kPoles && disp) {
            const Dom<T>& d = doms[c.dom];
            eb = (T(1) / ie - d.G) / S * F;
            for (int p = 0; p < d.npole; ++p) {
                T* pp = d.aade + ((long long)(a * d.npole + p) * 2 + 0) * d.bcell + bo;
                T* pq = pp + d.bcell;
                const T xp = *pp, xq = *pq;
                eb += d.g0[p] * xp + d.g1[p] * xq;
                *pp = d.M00[p] * xp + d.M10[p] * xq + (T(1) - d.M00[p]) / S * F;
                *pq = d.M01[p] * xp + d.M11[p] * xq - d.M01[p] / S * F;
            }
        } else {
            eb = F * recip_t(S * ie);
        }
        for (int s2 = 0; s2 < 2; ++s2) {
            const int ax = (a + 1 + s2) % 3;
            if (sl[ax] < 0) continue;
            T* p = c.apsiE[a][s2] + slab_off_c(c.n, c.ns, ax, i, j, k, sl[ax]);
            *p = c.cE[ax][x[ax]] * (*p + (s2 == 0 ? F : -F));
        }
        c.A[a][id] = eb;
    }
}

template <typename T>
void launch_adj_flush_cell(const Launch& L, const AdjCellArgs<T>& c, const Dom<T>* doms, T S, int poles,
                           int tensor) {
    const dim3 g((unsigned)((c.n[0] + kTileX - 1) / kTileX), (unsigned)((c.n[1] + kTileY - 1) / kTileY),
                 (unsigned)c.n[2]);
    if (tensor)
        k_adj_flush_cell<T, false, true><<<g, dim3(kTileX, kTileY), 0, L.stream>>>(c, doms, S);
    else if (poles)
        k_adj_flush_cell<T, true><<<g, dim3(kTileX, kTileY), 0, L.stream>>>(c, doms, S);
    else
        k_adj_flush_cell<T, false><<<g, dim3(kTileX, kTileY), 0, L.stream>>>(c, doms, S);
    ++*L.counter;
}

// Cells per thread of the transposed group kernels: the longest group that divides the rows and to which every array
// they access by groups is aligned.
template <typename T>
int adj_group(const AdjCellArgs<T>& c) {
    int v = sizeof(T) == 4 ? kAdjLong : 1;
    while (v > 1 && c.n[0] % v) v /= 2;
    auto fits = [&](const void* p) {
        while (v > 1 && (uintptr_t)p % (v * sizeof(T))) v /= 2;
    };
    for (const T* p : c.A) fits(p);
    for (const T* p : c.ie) fits(p);
    for (int q = 1; q < 3; ++q) {   // the memories along y and z
        fits(c.apsiE[(q + 1) % 3][1]);
        fits(c.apsiE[(q + 2) % 3][0]);
        fits(c.apsiH[(q + 1) % 3][1]);
        fits(c.apsiH[(q + 2) % 3][0]);
    }
    return v;
}

// ... and of these the length for the planes: shorter groups leave room for more blocks, which pays where the planes of small
// blocks do not find room at once (a step of 8 x 8 x 4096 13.4 -> 11.3 us; of 8 x 8 x 256, where one cell a thread has the
// longer way through its spills, 5.8 -> 6.3).
template <typename T>
int adj_length(const AdjCellArgs<T>& c) {
    const int v = adj_group(c);
    return c.n[2] > 152 * adj_group_blocks<T, kAdjLong>() ? plane_group((long long)c.n[0] * c.n[1], v) : v;
}

// The regions of the group kernels for groups of v cells, from the plain ranges [lo, hi) per axis (global planes along
// z); the grid.
template <typename T>
dim3 set_adj_regions(AdjCellArgs<T>& c, int v, const int* lo, const int* hi) {
    const int g = v < kAdjShort ? v : kAdjShort;
    c.gx = (lo[0] + v - 1) / v * v;
    c.gxn = std::max(0, hi[0] / v * v - c.gx);
    // a plane that fits one block as a whole is one region (its slab columns apart would take a second and a third block)
    if (c.gxn < c.n[0] && (long long)(c.n[0] / g) * c.n[1] <= kCellThreads) c.gxn = 0;
    if (c.gxn == 0) c.gx = c.n[0];   // every column belongs to region 1
    c.gy0 = std::min(lo[1], c.n[1]);
    c.gy1 = std::max(c.gy0, hi[1]);
    c.gz0 = lo[2];
    c.gz1 = std::max(lo[2], hi[2]);
    const int inner = c.gy1 - c.gy0;
    c.rows[0] = make_rows((unsigned)(c.gxn / v), inner);
    c.rows[1] = make_rows((unsigned)((c.n[0] - c.gxn) / g), c.n[1]);
    c.rows[2] = make_rows((unsigned)(c.gxn / g), c.n[1] - inner);
    c.nball = make_rows((unsigned)(c.gxn / g), c.n[1]).nb;
    const unsigned plain = c.rows[0].nb + c.rows[2].nb;
    return dim3(c.rows[1].nb + std::max(plain, c.nball), (unsigned)c.n[2]);
}

// The box [wlo, whi) of the cells that need the heavy kernel (poles, material cotangent), rounded out to its 16 x 16
// blocks (so that no group of cells straddles it); false if there are none.
template <typename T>
bool heavy_box(AdjCellArgs<T>& c, int poles) {
    bool any = false;
    auto join = [&](const int* lo, const int* hi) {
        if (hi[0] <= lo[0] || hi[1] <= lo[1] || hi[2] <= lo[2]) return;
        for (int q = 0; q < 3; ++q) {
            c.wlo[q] = any ? std::min(c.wlo[q], lo[q]) : lo[q];
            c.whi[q] = any ? std::max(c.whi[q], hi[q]) : hi[q];
        }
        any = true;
    };
    for (int q = 0; q < 3; ++q) c.wlo[q] = c.whi[q] = 0;
    if (poles) join(c.plo, c.phi);
    if (c.grad) join(c.glo, c.ghi);
    for (int q = 0; q < 2; ++q) {
        c.wlo[q] = c.wlo[q] / 16 * 16;
        c.whi[q] = std::min((c.whi[q] + 15) / 16 * 16, c.n[q]);
    }
    return any;
}

// The transposed E step of a domain: the group kernel over every cell outside the heavy box, then the heavy kernel over
// the box (they touch disjoint cells).  Compiled with the FP64 material cotangent or the poles, the kernel has half
// the occupancy: over a whole 256^3 domain with a 128 x 128 x 32 design box it took 323 us, 161 without.
template <typename T>
void launch_adj_e_cell(const Launch& L, const AdjCellArgs<T>& c0, const Dom<T>* doms, const Mon* mons, T S, int m,
                       int pending, int poles, int mon, int pole_grad, int tensor) {
    AdjCellArgs<T> c = c0;
    const dim3 b(kTileX, kTileY);
    auto grid = [&] {
        return dim3((unsigned)((c.whi[0] - c.wlo[0] + 15) / 16), (unsigned)((c.whi[1] - c.wlo[1] + 15) / 16),
                    (unsigned)(c.whi[2] - c.wlo[2]));
    };
    if (tensor) {
        // a tensor domain has no poles; its material cotangent comes from launch_tensor_grad
        for (int q = 0; q < 3; ++q) {
            c.wlo[q] = 0;
            c.whi[q] = c.n[q];
        }
        if (mon)
            launch_k(L, k_adj_e_cell<T, false, false, true, 0, true>, grid(), b, c, doms, mons, S, m, pending);
        else
            launch_k(L, k_adj_e_cell<T, false, false, false, 0, true>, grid(), b, c, doms, mons, S, m, pending);
        ++*L.counter;
        return;
    }
    const bool heavy = heavy_box(c, poles);
    const int v = adj_length(c);
    const dim3 gg = set_adj_regions(c, v, c.elo, c.ehi);
    with_group<T>(v, [&](auto V) {
        with_bool(c.ie[1] != c.ie[0] || c.ie[2] != c.ie[0], [&](auto A) {
            with_bool(mon, [&](auto M) {
                constexpr int kG = V() < kAdjShort ? V() : kAdjShort;
                launch_k(L, k_adj_e_group<T, V(), kG, A(), M()>, gg, dim3(kCellThreads), c, S, pending);
            });
        });
    });
    ++*L.counter;
    if (!heavy) return;
    const dim3 g = grid();
    with_bool(poles, [&](auto P) {
        with_bool(c.grad != nullptr, [&](auto D) {
            with_bool(mon, [&](auto M) {
                if constexpr (P()) {
                    if (pole_grad) {
                        if (pole_grad == 2)   // of two poles
                            launch_k(L, k_adj_e_cell<T, true, D(), M(), 2>, g, b, c, doms, mons, S, m, pending);
                        else
                            launch_k(L, k_adj_e_cell<T, true, D(), M(), 1>, g, b, c, doms, mons, S, m, pending);
                        return;
                    }
                }
                if constexpr (P() || D())
                    launch_k(L, k_adj_e_cell<T, P(), D(), M(), 0>, g, b, c, doms, mons, S, m, pending);
            });
        });
    });
    ++*L.counter;
}

template <typename T>
void launch_adj_h_cell(const Launch& L, const AdjCellArgs<T>& c0, T S, int m, int mon) {
    AdjCellArgs<T> c = c0;
    const int v = adj_length(c);
    // (region 0 must avoid PEC-held nodes too: the plain range starts past plane 0, see make_adj_args)
    const dim3 gg = set_adj_regions(c, v, c.hlo, c.hhi);
    with_group<T>(v, [&](auto V) {
        with_bool(mon, [&](auto M) {
            constexpr int kG = V() < kAdjShort ? V() : kAdjShort;
            launch_k(L, k_adj_h_group<T, V(), kG, M()>, gg, dim3(kCellThreads), c, S, m);
        });
    });
    ++*L.counter;
}

template <typename T>
void launch_adj_e(const Launch& L, const Dom<T>* doms, const Mon* mons, const Tile* tiles, int ntiles, T S, int m,
                  int pending, int general, int aniso, int pole_grad) {
    if (ntiles <= 0) return;
    const dim3 b(kTileX, kTileY);
    if (general && pole_grad)
        k_adj_e_gen<T, true><<<ntiles, b, 0, L.stream>>>(doms, mons, tiles, S, m, pending);
    else if (general)
        k_adj_e_gen<T, false><<<ntiles, b, 0, L.stream>>>(doms, mons, tiles, S, m, pending);
    else if (aniso)
        k_adj_e_int<T, true><<<ntiles, b, 0, L.stream>>>(doms, mons, tiles, S, m, pending);
    else
        k_adj_e_int<T, false><<<ntiles, b, 0, L.stream>>>(doms, mons, tiles, S, m, pending);
    ++*L.counter;
}

template <typename T>
void launch_adj_h(const Launch& L, const Dom<T>* doms, const Mon* mons, const Tile* tiles, int ntiles, T S, int m,
                  int general) {
    if (ntiles <= 0) return;
    const dim3 b(kTileX, kTileY);
    if (general)
        k_adj_h_gen<T><<<ntiles, b, 0, L.stream>>>(doms, mons, tiles, S, m);
    else
        k_adj_h_int<T><<<ntiles, b, 0, L.stream>>>(doms, mons, tiles, S, m);
    ++*L.counter;
}

template <typename T>
void launch_adj_flush(const Launch& L, const Dom<T>* doms, const Tile* tiles, int ntiles, T S) {
    if (ntiles <= 0) return;
    k_adj_flush<T><<<ntiles, dim3(kTileX, kTileY), 0, L.stream>>>(doms, tiles, S);
    ++*L.counter;
}

template <typename T>
void launch_inject_box(const Launch& L, const Dom<T>* dom, const Mon* mons, const int* lo, const int* hi,
                       long long pidx_e, long long pidx_h, T* inj) {
    const long long vol = (long long)(hi[0] - lo[0]) * (hi[1] - lo[1]) * (hi[2] - lo[2]);
    if (vol <= 0) return;
    const int bs = 256;
    k_inject_box<T><<<(unsigned)((vol + bs - 1) / bs), bs, 0, L.stream>>>(dom, mons, make_int3(lo[0], lo[1], lo[2]),
                                                                           make_int3(hi[0], hi[1], hi[2]), pidx_e,
                                                                           pidx_h, inj);
    ++*L.counter;
}

template <typename T>
void launch_inject(const Launch& L, const Dom<T>* doms, const Mon* mons, const int* entries, int nentries,
                   long long nthreads, const long long* entry_begin, int step, int kind) {
    if (nentries <= 0 || nthreads <= 0) return;
    const int bs = 256;
    k_inject<T><<<(unsigned)((nthreads + bs - 1) / bs), bs, 0, L.stream>>>(doms, mons, entries, nentries, nthreads,
                                                                           entry_begin, step, kind);
    ++*L.counter;
}

#define GBFDTD_INST(T)                                                                                          \
    template void launch_adj_e<T>(const Launch&, const Dom<T>*, const Mon*, const Tile*, int, T, int, int, int, \
                                  int, int);                                                                    \
    template void launch_adj_h<T>(const Launch&, const Dom<T>*, const Mon*, const Tile*, int, T, int, int);     \
    template void launch_adj_flush<T>(const Launch&, const Dom<T>*, const Tile*, int, T);                       \
    template void launch_inject<T>(const Launch&, const Dom<T>*, const Mon*, const int*, int, long long,        \
                                   const long long*, int, int);                                                 \
    template void launch_inject_box<T>(const Launch&, const Dom<T>*, const Mon*, const int*, const int*,         \
                                       long long, long long, T*);                                               \
    template void launch_adj_e_cell<T>(const Launch&, const AdjCellArgs<T>&, const Dom<T>*, const Mon*, T, int,  \
                                       int, int, int, int, int);                                                \
    template void launch_adj_h_cell<T>(const Launch&, const AdjCellArgs<T>&, T, int, \
                                       int);                                                                    \
    template void launch_adj_flush_cell<T>(const Launch&, const AdjCellArgs<T>&, const Dom<T>*, T, int, int);
GBFDTD_INST(float)
GBFDTD_INST(double)
#undef GBFDTD_INST

}  // namespace gbfdtd
