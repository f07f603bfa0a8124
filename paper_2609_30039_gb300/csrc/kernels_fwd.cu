// Forward half-steps of the Yee leapfrog (arxiv 2609.30039, Sec. 2.1 Eq. (yee)) with the CPML
// memories of Sec. 2.2, the trapezoidal Drude/Lorentz update and diagonal eps^-1 of Sec. 2.3,
// soft sources and running DFT monitors of Sec. 2.4.
//
// Two work decompositions of a half-step: the tile kernels (mode 0), where a tile is 32 x 8 columns of
// one domain and each thread owns a column (i, j) and marches k over the tile's z range; and the per-cell
// kernels (mode 4, below), where every cell of a domain is in one launch and a thread updates a group of
// cells of a row.  Both give the same bits; the tile kernels also serve as the check of the others.
#include <algorithm>
#include <type_traits>

#include "fdtd_internal.cuh"

namespace gbfdtd {

// CPML coefficients of one node along one axis: y = D/kappa + psi, psi <- b psi + c D.
template <typename T>
struct Cpml1 {
    int s;        // slab index, -1 outside the slabs
    T b, c, k;
};

template <typename T>
__device__ __forceinline__ Cpml1<T> cpml_at(const Dom<T>& d, const T* coef, int q, int x) {
    Cpml1<T> r;
    r.s = d.ns[q] ? slab_of(x, d.dlo[q], d.dhi[q], d.n[q]) : -1;
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

// In-slab CPML correction of one derivative: psi <- b psi + c D first, then y = D/kappa + psi
// (c D rounded, then two fused multiply-adds).

template <typename T>
__device__ __forceinline__ T cpml_rec(T b, T c, T kinv, T* psi, T D) {
    const T cd = c * D;
    const T ps = fma_t(b, *psi, cd);
    *psi = ps;
    return fma_t(kinv, D, ps);
}

template <typename T>
__device__ __forceinline__ T cpml_apply(const Cpml1<T>& q, T* psi, T D) {
    return cpml_rec(q.b, q.c, q.k, psi, D);
}

// Trapezoidal pole update of one E component (Sec. 2.3):
// (eps_inf + G) E^{n+1} = (eps_inf + G) E^n + Delta,
// Delta = S curl + sum_p (P_p - (M_p x_p)_P - 2 g_p E^n);  x_p <- M_p x_p + g_p (E^{n+1} + E^n).
// (Multiply-adds are written as explicit fused operations so every kernel rounds alike.)
template <typename T>
__device__ __forceinline__ T ade_update(const Dom<T>& d, int a, long long bo, T e0, T ie, T scurl) {
    T delta = scurl;
    T* base = d.ade + (long long)a * d.npole * 2 * d.bcell + bo;
    for (int p = 0; p < d.npole; ++p) {
        const T P = base[(2 * p) * d.bcell], Q = base[(2 * p + 1) * d.bcell];
        const T mp = fma_t(d.M00[p], P, d.M01[p] * Q);
        delta = delta + fma_t(-T(2) * d.g0[p], e0, P - mp);
    }
    const T e1 = fma_t(ie / fma_t(ie, d.G, T(1)), delta, e0);
    const T es = e1 + e0;
    for (int p = 0; p < d.npole; ++p) {
        T* pp = base + (2 * p) * d.bcell;
        T* pq = base + (2 * p + 1) * d.bcell;
        const T P = *pp, Q = *pq;
        *pp = fma_t(d.g0[p], es, fma_t(d.M00[p], P, d.M01[p] * Q));
        *pq = fma_t(d.g1[p], es, fma_t(d.M10[p], P, d.M11[p] * Q));
    }
    return e1;
}

template <typename T>
__device__ __forceinline__ T src_add(const Dom<T>& d, const Src* __restrict__ srcs, int comp, int i, int j, int k,
                                     int step) {
    return src_add_t<T>(d, srcs, comp, i, j, k, step);
}

// Running DFT (Sec. 2.4), F += f exp(i w t) accumulated in FP64, of one work item: up to 256
// consecutive cells of one monitor (one per thread), for the recorded components of one kind
// (0: E at t = n+1, 1: H at t = n+3/2).  It runs beside the field updates, never on their
// critical path: the E part of step n while H is updated, the H part while E of step n+1 is (each
// only reads the field the other half-step leaves alone).  A cell's accumulators are updated in
// batches of four, loads before stores, one memory round trip per batch.
template <typename T>
__device__ __forceinline__ void dft_item(const Dom<T>* __restrict__ doms, const Mon* __restrict__ mons,
                                         const DftItem& it, int kind, int step) {
    const Mon& m = mons[it.mon];
    const long long cell = it.begin + threadIdx.y * kTileX + threadIdx.x;
    if (cell >= it.end) return;
    const int i = m.lo[0] + (int)(cell % m.bx);
    const int j = m.lo[1] + (int)((cell / m.bx) % m.by);
    const int k = m.lo[2] + (int)(cell / ((long long)m.bx * m.by)) - it.kz0;
    const Dom<T>& d = doms[it.dom];
    const long long id = cidx(d.n, i, j, k);
    const double2* ph = m.phase + ((long long)step * 2 + kind) * m.nf;
    const int nf = m.nf;
    int ci = 0;
    for (int c = 0; c < 6; ++c) {
        if (!((m.mask >> c) & 1u)) continue;
        if (c / 3 == kind) {
            const double v = (double)d.F[c][id];
            double2* acc = m.acc + (long long)ci * nf * m.ncell + cell;
            for (int f0 = 0; f0 < nf; f0 += 4) {
                double2 x[4], p[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int f = f0 + q < nf ? f0 + q : f0;
                    x[q] = acc[(long long)f * m.ncell];
                    p[q] = ph[f];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (f0 + q >= nf) break;
                    x[q].x = fma_t(v, p[q].x, x[q].x);
                    x[q].y = fma_t(v, p[q].y, x[q].y);
                    acc[(long long)(f0 + q) * m.ncell] = x[q];
                }
            }
        }
        ++ci;
    }
}

// Per-half-step DFT launch: one block per work item; the step is *d_base + offset (the first
// step of the launched batch plus this launch's position in it, so a captured graph replays).
template <typename T>
__global__ void __launch_bounds__(kTileX* kTileY)
    k_dft(const Dom<T>* __restrict__ doms, const Mon* __restrict__ mons, const DftItem* __restrict__ items, int kind,
          const int* __restrict__ d_base, int offset) {
    dft_item(doms, mons, items[blockIdx.x], kind, *d_base + offset);
}

// DFT of steps t0 .. cnt - 1 of a batch from the monitor rings (per-cell mode): block (x, y) takes work item
// x for the monitor's y-th component (one thread per monitor cell), so the FP64 work of a batch
// spreads over items x components blocks; each accumulator takes the samples of steps base,
// base + 1, ... in order with the fused multiply-adds of dft_item, so it ends bit for bit where cnt
// per-step launches of each kind would leave it, with one accumulator load and store per batch
// instead of per step.
template <typename T>
__global__ void __launch_bounds__(kTileX* kTileY)
    k_dft_ring(const Mon* __restrict__ mons, const DftItem* __restrict__ items, const int* __restrict__ d_base, int t0,
               int cnt) {
    const DftItem& it = items[blockIdx.x];
    const Mon& m = mons[it.mon];
    const int ci = blockIdx.y;
    const long long cell = it.begin + threadIdx.y * kTileX + threadIdx.x;
    if (ci >= m.ncomp || cell >= it.end) return;
    const int base = *d_base, nf = m.nf;
    const long long slot = (long long)m.ncomp * m.ncell;
    {
        const int kind = m.comps[ci] >= 3 ? 1 : 0;
        const T* r = (const T*)m.ring + (long long)ci * m.ncell + cell;
        double2* acc = m.acc + (long long)ci * nf * m.ncell + cell;
        for (int f0 = 0; f0 < nf; f0 += 4) {
            double2 x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = acc[(long long)(f0 + q < nf ? f0 + q : f0) * m.ncell];
            for (int t = t0; t < cnt; ++t) {
                const double v = (double)r[t * slot];
                const double2* ph = m.phase + ((long long)(base + t) * 2 + kind) * nf + f0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (f0 + q >= nf) break;
                    const double2 p = ph[q];
                    x[q].x = fma_t(v, p.x, x[q].x);
                    x[q].y = fma_t(v, p.y, x[q].y);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (f0 + q >= nf) break;
                acc[(long long)(f0 + q) * m.ncell] = x[q];
            }
        }
    }
}

// Monitor samples: plane kg (global; block-uniform in the per-cell kernels) crosses the domain's
// monitor box and the step stores samples, then cell (i, j) lies in the box; the sample of a
// component goes to slot a.offset of its ring at sample_off.
template <typename T>
__device__ __forceinline__ bool in_sample_plane(const CellArgs<T>& c, const StepArgs& a, int kg) {
    return (unsigned)(kg - c.slo[2]) < (unsigned)(c.shi[2] - c.slo[2]) && a.ring;
}
template <typename T>
__device__ __forceinline__ bool in_sample_rect(const CellArgs<T>& c, int i, int j) {
    return (unsigned)(i - c.slo[0]) < (unsigned)(c.shi[0] - c.slo[0]) &&
           (unsigned)(j - c.slo[1]) < (unsigned)(c.shi[1] - c.slo[1]);
}
template <typename T>
__device__ __forceinline__ long long sample_off(const CellArgs<T>& c, const StepArgs& a, int i, int j, int kg) {
    return (long long)a.offset * c.sstride +
           ((long long)(kg - c.slo[2]) * (c.shi[1] - c.slo[1]) + (j - c.slo[1])) * (c.shi[0] - c.slo[0]) +
           (i - c.slo[0]);
}

__global__ void k_copy_int(const int* __restrict__ src, int* __restrict__ dst) { *dst = *src; }

__global__ void k_set_int(int* __restrict__ dst, int v) { *dst = v; }

// Blocks per SM the per-launch kernels are compiled for.  Interior tiles run the plain register
// path at full occupancy (8 blocks of 256 threads in FP32, at most 32 registers): the warps in
// flight are what keeps enough loads outstanding to approach the DRAM bandwidth.
#ifndef GBFDTD_INT_BLOCKS_F32
#define GBFDTD_INT_BLOCKS_F32 8
#endif
template <typename T>
constexpr int min_blocks(bool general) {
    return general ? (sizeof(T) == 4 ? 4 : 2) : (sizeof(T) == 4 ? GBFDTD_INT_BLOCKS_F32 : 4);
}

// E half-step (Eq. (yee) first half) of a tile.  kGen = false: the tile touches no CPML slab,
// PEC plane, domain edge or dispersive cell, so none of that code is compiled in.  Every load of
// a plane is issued before any store of it; H_x, H_y of plane k-1 stay in registers.
template <typename T, bool kGen, bool kAniso>
__device__ __forceinline__ void tile_e(const Dom<T>* __restrict__ doms, const Tile& t, T S, const StepArgs& a,
                                       int step) {
    const Dom<T>& d = doms[t.dom];
    const int nx = d.n[0], ny = d.n[1];
    int i, j;
    tile_coords(t, i, j);
    if (i < 0 || j < 0) return;
    const bool fsrc = t.flags & kTileSrcE;
    const long long nxy = (long long)nx * ny;
    T* Ex = d.F[0];
    T* Ey = d.F[1];
    T* Ez = d.F[2];
    const T* Hx = d.F[3];
    const T* Hy = d.F[4];
    const T* Hz = d.F[5];
    const T* ie0 = d.ie[0];
    const T* ie1 = d.ie[1];
    const T* ie2 = d.ie[2];
    Cpml1<T> cx, cy;
    bool pi = false, pj = false;              // PEC plane at this column's x / y
    bool hasx = true, hasy = true;            // the -x / -y neighbour exists (wraps if periodic)
    long long oxm = -1, oym = -(long long)nx;
    if (kGen) {
        cx = cpml_at(d, d.cE[0], 0, i);
        cy = cpml_at(d, d.cE[1], 1, j);
        pi = i == 0 && !d.per[0];
        pj = j == 0 && !d.per[1];
        oxm = nb_minus(i, nx, 1, d.per[0], &hasx);
        oym = nb_minus(j, ny, nx, d.per[1], &hasy);
    }
    long long id = (long long)t.z0 * nxy + (long long)j * nx + i;
    T hxz = T(0), hyz = T(0);
    if (!kGen || t.z0 > 0) {
        hxz = Hx[id - nxy];
        hyz = Hy[id - nxy];
    }
    for (int k = t.z0; k < t.z1; ++k, id += nxy) {
        const T hx = Hx[id], hy = Hy[id], hz = Hz[id];
        const T hz_ym = (!kGen || hasy) ? Hz[id + oym] : T(0);
        const T hx_ym = (!kGen || hasy) ? Hx[id + oym] : T(0);
        const T hz_xm = (!kGen || hasx) ? Hz[id + oxm] : T(0);
        const T hy_xm = (!kGen || hasx) ? Hy[id + oxm] : T(0);
        T ex = Ex[id], ey = Ey[id], ez = Ez[id];
        const T iex = ie0[id];
        const T iey = kAniso ? ie1[id] : iex;
        const T iez = kAniso ? ie2[id] : iex;
        T yx1 = hz - hz_ym, yx2 = hy - hyz;  // Ex: dHz/dy, dHy/dz
        T yy1 = hx - hxz, yy2 = hz - hz_xm;  // Ey: dHx/dz, dHz/dx
        T yz1 = hy - hy_xm, yz2 = hx - hx_ym;  // Ez: dHy/dx, dHx/dy
        hxz = hx;
        hyz = hy;
        if (kGen) {
            const bool pk = k == 0;
            const bool px = pj || pk, py = pi || pk, pz = pi || pj;  // PEC-held components
            const Cpml1<T> cz = cpml_at(d, d.cE[2], 2, k);
            if (cz.s >= 0) {
                const long long o = ((long long)cz.s * ny + j) * nx + i;
                if (!px) yx2 = cpml_apply(cz, d.psiE[0][1] + o, yx2);
                if (!py) yy1 = cpml_apply(cz, d.psiE[1][0] + o, yy1);
            }
            if (cx.s >= 0) {
                const long long o = ((long long)k * ny + j) * d.ns[0] + cx.s;
                if (!py) yy2 = cpml_apply(cx, d.psiE[1][1] + o, yy2);
                if (!pz) yz1 = cpml_apply(cx, d.psiE[2][0] + o, yz1);
            }
            if (cy.s >= 0) {
                const long long o = ((long long)k * d.ns[1] + cy.s) * nx + i;
                if (!px) yx1 = cpml_apply(cy, d.psiE[0][0] + o, yx1);
                if (!pz) yz2 = cpml_apply(cy, d.psiE[2][1] + o, yz2);
            }
            const bool disp = d.npole > 0 && i >= d.blo[0] && i < d.bhi[0] && j >= d.blo[1] && j < d.bhi[1] &&
                              k >= d.blo[2] && k < d.bhi[2] && d.mask[id];
            if (disp) {
                const long long bo = ade_off(d, i, j, k);
                if (!px) ex = ade_update(d, 0, bo, ex, iex, S * (yx1 - yx2));
                if (!py) ey = ade_update(d, 1, bo, ey, iey, S * (yy1 - yy2));
                if (!pz) ez = ade_update(d, 2, bo, ez, iez, S * (yz1 - yz2));
            } else {
                if (!px) ex = fma_t(S * iex, (yx1 - yx2), ex);
                if (!py) ey = fma_t(S * iey, (yy1 - yy2), ey);
                if (!pz) ez = fma_t(S * iez, (yz1 - yz2), ez);
            }
            // a PEC-held component keeps its (zero) value and receives no source
        } else {
            ex = fma_t(S * iex, (yx1 - yx2), ex);
            ey = fma_t(S * iey, (yy1 - yy2), ey);
            ez = fma_t(S * iez, (yz1 - yz2), ez);
        }
        if (fsrc) {
            ex += src_add(d, a.srcs, 0, i, j, k, step);
            ey += src_add(d, a.srcs, 1, i, j, k, step);
            ez += src_add(d, a.srcs, 2, i, j, k, step);
        }
        if (kGen) {
            const bool pk = k == 0;
            if (!(pj || pk)) Ex[id] = ex;
            if (!(pi || pk)) Ey[id] = ey;
            if (!(pi || pj)) Ez[id] = ez;
        } else {
            Ex[id] = ex;
            Ey[id] = ey;
            Ez[id] = ez;
        }
    }
}

template <typename T, bool kGen, bool kAniso>
__global__ void __launch_bounds__(kTileX* kTileY, min_blocks<T>(kGen))
    k_e_update(const Dom<T>* __restrict__ doms, const Tile* __restrict__ tiles, T S, const StepArgs a) {
    tile_e<T, kGen, kAniso>(doms, tiles[blockIdx.x], S, a, *a.d_step);
}

// H half-step (Eq. (yee) second half) of a tile; E_x, E_y of plane k+1 are carried to the next
// plane in registers.  kEnergy adds W_{n+1} = 1/2 sum eps |E|^2 + 1/2 sum H^{n+1/2} H^{n+3/2}.
template <typename T, bool kGen, bool kEnergy>
__device__ __forceinline__ void tile_h(const Dom<T>* __restrict__ doms, const Tile& t, T S, const StepArgs& a,
                                       int step) {
    const Dom<T>& d = doms[t.dom];
    const int nx = d.n[0], ny = d.n[1], nz = d.n[2];
    int i, j;
    tile_coords(t, i, j);
    const bool fsrc = t.flags & kTileSrcH;
    double w = 0.0;
    if (i >= 0 && j >= 0) {
        const long long nxy = (long long)nx * ny;
        const T* Ex = d.F[0];
        const T* Ey = d.F[1];
        const T* Ez = d.F[2];
        T* Hx = d.F[3];
        T* Hy = d.F[4];
        T* Hz = d.F[5];
        Cpml1<T> cx, cy;
        bool xe = true, ye = true;  // the +x / +y neighbour node exists (wraps if periodic)
        long long oxp = 1, oyp = nx;
        if (kGen) {
            cx = cpml_at(d, d.cH[0], 0, i);
            cy = cpml_at(d, d.cH[1], 1, j);
            oxp = nb_plus(i, nx, 1, d.per[0], &xe);
            oyp = nb_plus(j, ny, nx, d.per[1], &ye);
        }
        long long id = (long long)t.z0 * nxy + (long long)j * nx + i;
        T exk = Ex[id], eyk = Ey[id];
        for (int k = t.z0; k < t.z1; ++k, id += nxy) {
            const bool ze = !kGen || k + 1 < nz;
            const T exn = ze ? Ex[id + nxy] : T(0);
            const T eyn = ze ? Ey[id + nxy] : T(0);
            const T ez = Ez[id];
            const T ez_yp = ye ? Ez[id + oyp] : T(0);
            const T ez_xp = xe ? Ez[id + oxp] : T(0);
            const T ey_xp = xe ? Ey[id + oxp] : T(0);
            const T ex_yp = ye ? Ex[id + oyp] : T(0);
            const T hx = Hx[id], hy = Hy[id], hz = Hz[id];
            T yx1 = ez_yp - ez, yx2 = eyn - eyk;  // Hx: dEz/dy, dEy/dz
            T yy1 = exn - exk, yy2 = ez_xp - ez;  // Hy: dEx/dz, dEz/dx
            T yz1 = ey_xp - eyk, yz2 = ex_yp - exk;  // Hz: dEy/dx, dEx/dy
            if (kGen) {
                const Cpml1<T> cz = cpml_at(d, d.cH[2], 2, k);
                if (cz.s >= 0) {
                    const long long o = ((long long)cz.s * ny + j) * nx + i;
                    yx2 = cpml_apply(cz, d.psiH[0][1] + o, yx2);
                    yy1 = cpml_apply(cz, d.psiH[1][0] + o, yy1);
                }
                if (cx.s >= 0) {
                    const long long o = ((long long)k * ny + j) * d.ns[0] + cx.s;
                    yy2 = cpml_apply(cx, d.psiH[1][1] + o, yy2);
                    yz1 = cpml_apply(cx, d.psiH[2][0] + o, yz1);
                }
                if (cy.s >= 0) {
                    const long long o = ((long long)k * d.ns[1] + cy.s) * nx + i;
                    yx1 = cpml_apply(cy, d.psiH[0][0] + o, yx1);
                    yz2 = cpml_apply(cy, d.psiH[2][1] + o, yz2);
                }
            }
            T hx1 = fma_t(-S, (yx1 - yx2), hx);
            T hy1 = fma_t(-S, (yy1 - yy2), hy);
            T hz1 = fma_t(-S, (yz1 - yz2), hz);
            if (fsrc) {
                hx1 += src_add(d, a.srcs, 3, i, j, k, step);
                hy1 += src_add(d, a.srcs, 4, i, j, k, step);
                hz1 += src_add(d, a.srcs, 5, i, j, k, step);
            }
            Hx[id] = hx1;
            Hy[id] = hy1;
            Hz[id] = hz1;
            if (kEnergy) {
                w += 0.5 * ((double)hx * hx1 + (double)hy * hy1 + (double)hz * hz1);
                w += 0.5 * ((double)exk * exk / (double)d.ie[0][id] + (double)eyk * eyk / (double)d.ie[1][id] +
                            (double)ez * ez / (double)d.ie[2][id]);
            }
            exk = exn;
            eyk = eyn;
        }
    }
    if (kEnergy) {
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        if ((threadIdx.x & 31) == 0 && d.energy && step < d.energy_cap) atomicAdd(d.energy + step, w);
    }
}

template <typename T, bool kGen, bool kEnergy>
__global__ void __launch_bounds__(kTileX* kTileY, min_blocks<T>(kGen))
    k_h_update(const Dom<T>* __restrict__ doms, const Tile* __restrict__ tiles, T S, const StepArgs a,
               unsigned advance_blocks) {
    const int step = *a.d_step;
    tile_h<T, kGen, kEnergy>(doms, tiles[blockIdx.x], S, a, step);
    if (advance_blocks) {
        // the H launches of a step (general and interior, possibly running concurrently) hold
        // advance_blocks blocks together; the last of them to finish advances the device step
        // counter (every block has read it)
        __syncthreads();
        if (threadIdx.x == 0 && threadIdx.y == 0) {
            __threadfence();
            const unsigned done = atomicAdd(a.d_ticket, 1u);
            if (done == advance_blocks - 1) {
                *a.d_ticket = 0u;
                *a.d_step = step + 1;
                __threadfence();
            }
        }
    }
}

// ---- per-cell streaming kernels -------------------------------------------------------------
// Every cell of a domain in one launch, no z-march and no tile classes.  A thread updates kV consecutive
// cells of a row (four in FP32 where the row length and the arrays' alignment allow it, else two or
// one): the groups of a plane are numbered through its rows, so no lane is left over at a row's end, and the
// -1 / +1 neighbours along x are the thread's own cells or the neighbouring lane's (a shuffle; one scalar load
// at a warp's or row's edge).  All loads of a thread are independent (the z-1 / z+1 neighbour comes from L2)
// and the domain's pointers arrive as a kernel parameter, so the first loads issue at once.
// What bounds it: with one cell per thread, instruction issue as much as memory (234 / 198 executed instructions
// per cell for E / H at 128^3 with 10-cell CPML, issue slots 74% busy); a group of four cells shares the index,
// address, CPML and PEC work.  Measured per step (E + H launches): 128^3 with CPML 34.9 -> 23.1 us, without CPML
// 16.5 us (state in L2: 10 TB/s of field traffic); 256^3 269 -> 206 us; 512^3 in whole passes 1971 -> 1594 us (E + H back to back 1521, 6.7 TB/s of
// algorithmic bytes, DRAM); 243 x 251 x 229 (one cell per thread) 245 -> 220 us.  Arithmetic per cell is the
// same as in tile_e / tile_h.
// Blocks per SM the kernels are compiled for (registers for all loads of a group in flight), as threads per SM.  FP32,
// four cells: 768 (80 registers; 512 and 1024 were slower: 256^3 206 against 236 and 272 us), two: 1024, one: 1536;
// poles: 512.  FP64 runs one cell per thread with 1024: the FP64 pipe bounds it, and pairs of cells only cost
// occupancy (128^3: 131 against 138 us a step).
template <typename T, int kV, bool kPoles = false>
constexpr int cell_blocks() {
    return (sizeof(T) == 4 ? (kPoles ? 512 : kV == 4 ? 768 : kV == 2 ? 1024 : 1536) : (kPoles ? 768 : 1024)) / kCellThreads;
}

// Cells per thread in the columns that hold x slabs, where the interior has v: two instead of four, which with the
// memories along x would need more registers than 768 threads per SM have (128^3 with blocks of 256: 25.5 us a
// step; four: 30.8, one: 28.2).
__host__ __device__ constexpr int edge_group(int v) { return v == 4 ? 2 : v; }

// The group of kV cells of this thread: row j, first cell i; left / right: whether the neighbouring lane holds the
// neighbouring group; live: the thread has a group (others run along on the last one, without effect).
struct GroupAt {
    int i, j;
    bool left, right, live;
};

// A plane is cut into two regions, each numbered row by row: the groups of a row that hold no cell of an x slab (the
// first rows[0].nb blocks), then those that do (kEdge), so that the work along x is that of whole warps instead of a few
// lanes of every warp (at 128^3 with 10-cell slabs every 128-cell warp row would hold some).  The quotient by the
// row length is a multiply by a host-computed reciprocal (exact for t < 2^31, see make_rows).
template <typename T, int kV, bool kEdge>
__device__ __forceinline__ GroupAt group_at(const CellArgs<T>& c, unsigned block) {
    const GroupRows& r = c.rows[kEdge ? 1 : 0];
    const unsigned n = r.gp * (unsigned)c.n[1];
    unsigned t = block * kCellThreads + threadIdx.x;
    GroupAt g;
    g.live = t < n;
    if (!g.live) t = n - 1;
    const unsigned row = group_row(r, t);
    const int col = (int)(t - row * r.gp), lane = threadIdx.x & 31;
    g.j = (int)row;
    const int x = col * kV;
    g.i = kEdge ? (x < c.xlo ? x : x + c.xin) : x + c.xlo;
    g.left = lane != 0 && col != 0 && !(kEdge && x == c.xlo);
    g.right = lane != 31 && col + 1 != (int)r.gp && !(kEdge && x + kV == c.xlo);
    return g;
}

// CPML memories of a group, loaded together with the fields (before anything waits for a load, so a slab cell costs
// one memory latency like any other): per axis the two memories along it.  Only edge groups lie in x slabs; where
// the memories' rows divide into groups (c.xvec) the group's ones are one vector (a group only partly in a slab
// loads a neighbour's along), else they are read cell by cell.
template <typename T, int kV, bool kEdge>
struct GroupCpml {
    int sy, sz;           // slab indices along y, z (-1: outside)
    unsigned sx;          // cells (bits) in an x slab
    bool xvec;
    unsigned ox, oy, oz;  // offsets in the memories (x: of the group's first cell)
    T by, cy, ky, bz, cz, kz;
    Group<T, kV> x0, x1, y0, y1, z0, z1;
};

template <typename T, int kV, bool kEdge>
__device__ __forceinline__ void load_cpml(const CellArgs<T>& c, int i, int j, int k, GroupCpml<T, kV, kEdge>& m) {
    const int nx = c.n[0], ny = c.n[1], kg = k + c.kz0;
    m.sz = c.ns[2] ? slab_of(kg, c.dlo[2], c.dhi[2], c.nzg) : -1;
    m.sy = c.ns[1] ? slab_of(j, c.dlo[1], c.dhi[1], ny) : -1;
    m.sx = 0;
    if (m.sz >= 0) {
        m.oz = ((unsigned)m.sz * ny + j) * nx + i;
        m.z0 = ld_group<T, kV>(c.psi[0][1] + m.oz);
        m.z1 = ld_group<T, kV>(c.psi[1][0] + m.oz);
        m.bz = c.coef[2][kg];
        m.cz = c.coef[2][c.nzg + kg];
        m.kz = c.coef[2][2 * c.nzg + kg];
    }
    if (m.sy >= 0) {
        m.oy = (unsigned)(k * c.ns[1] + m.sy) * nx + i;
        m.y0 = ld_group<T, kV>(c.psi[0][0] + m.oy);
        m.y1 = ld_group<T, kV>(c.psi[2][1] + m.oy);
        m.by = c.coef[1][j];
        m.cy = c.coef[1][ny + j];
        m.ky = c.coef[1][2 * ny + j];
    }
    if (kEdge && c.ns[0]) {
        const int hi = nx - c.dhi[0];   // first cell of the high slab
#pragma unroll
        for (int q = 0; q < kV; ++q)
            if (i + q < c.dlo[0] || i + q >= hi) m.sx |= 1u << q;
        // a group between the slabs of a narrow domain may hold cells of both: those are read one by one
        const bool low = i < c.dlo[0], both = low && i + kV > hi;
        m.xvec = c.xvec && !both;
        m.ox = (unsigned)(k * ny + j) * c.ns[0] + (unsigned)(low ? i : i - hi + c.dlo[0]);
        if (m.xvec) {
            if (m.sx) {
                m.x0 = ld_group<T, kV>(c.psi[1][1] + m.ox);
                m.x1 = ld_group<T, kV>(c.psi[2][0] + m.ox);
            }
        } else {
#pragma unroll
            for (int q = 0; q < kV; ++q)
                if (m.sx >> q & 1) {
                    const unsigned o = m.ox + q - (low && i + q >= hi ? (unsigned)(hi - c.dlo[0]) : 0u);
                    m.x0[q] = c.psi[1][1][o];
                    m.x1[q] = c.psi[2][0][o];
                }
        }
    }
}

// Advances the memories and corrects the derivatives: xa, xb along x (of components y, z), ya, yb along y (x, z),
// za, zb along z (x, y).  hx, hy, hz: cells (bits) whose component x, y, z is held: its memories stay.
template <typename T, int kV, bool kEdge>
__device__ __forceinline__ void apply_cpml(const CellArgs<T>& c, int i, GroupCpml<T, kV, kEdge>& m, Group<T, kV>& xa,
                                           Group<T, kV>& xb, Group<T, kV>& ya, Group<T, kV>& yb, Group<T, kV>& za,
                                           Group<T, kV>& zb, unsigned hx, unsigned hy, unsigned hz) {
    if (m.sz >= 0) {
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            if (!(hx >> q & 1)) za[q] = cpml_rec(m.bz, m.cz, m.kz, &m.z0[q], za[q]);
            if (!(hy >> q & 1)) zb[q] = cpml_rec(m.bz, m.cz, m.kz, &m.z1[q], zb[q]);
        }
        st_group(c.psi[0][1] + m.oz, m.z0);
        st_group(c.psi[1][0] + m.oz, m.z1);
    }
    if (kEdge && m.sx) {
        const int nx = c.n[0], hi = nx - c.dhi[0];
        const T* co = c.coef[0] + i;
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            if (!(m.sx >> q & 1)) continue;
            const T b = co[q], cc = co[nx + q], kk = co[2 * nx + q];
            if (!(hy >> q & 1)) xa[q] = cpml_rec(b, cc, kk, &m.x0[q], xa[q]);
            if (!(hz >> q & 1)) xb[q] = cpml_rec(b, cc, kk, &m.x1[q], xb[q]);
        }
        if (m.xvec && m.sx == (1u << kV) - 1) {
            st_group(c.psi[1][1] + m.ox, m.x0);
            st_group(c.psi[2][0] + m.ox, m.x1);
        } else {
#pragma unroll
            for (int q = 0; q < kV; ++q)
                if (m.sx >> q & 1) {
                    const unsigned o = m.ox + q - (i < c.dlo[0] && i + q >= hi ? (unsigned)(hi - c.dlo[0]) : 0u);
                    c.psi[1][1][o] = m.x0[q];
                    c.psi[2][0][o] = m.x1[q];
                }
        }
    }
    if (m.sy >= 0) {
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            if (!(hx >> q & 1)) ya[q] = cpml_rec(m.by, m.cy, m.ky, &m.y0[q], ya[q]);
            if (!(hz >> q & 1)) yb[q] = cpml_rec(m.by, m.cy, m.ky, &m.y1[q], yb[q]);
        }
        st_group(c.psi[0][0] + m.oy, m.y0);
        st_group(c.psi[2][1] + m.oy, m.y1);
    }
}

// Soft sources of components c0 .. c0 + 2 on a group whose cells meet the bounding box of the half-step's sources.
// The boxes come with the kernel's arguments: a sheet normal to x is met by some lane of every warp of its
// planes, so a walk through descriptors in memory there would cost every warp two more memory latencies.
template <typename T, int kV>
__device__ __forceinline__ void add_sources(const CellArgs<T>& c, const StepArgs& a, int c0, int i, int j, int kg,
                                            Group<T, kV>& v0, Group<T, kV>& v1, Group<T, kV>& v2) {
    const int step = *a.d_base + a.offset;
    Group<T, kV> s0{}, s1{}, s2{};
    for (int s = 0; s < c.nsb; ++s) {
        const SrcBox& b = c.sb[s];
        if (j < b.lo[1] || j >= b.hi[1] || kg < b.lo[2] || kg >= b.hi[2] || step >= b.n) continue;
        const T w = (T)b.wave[step];
        const int comp = b.comp - c0;
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const T x = i + q >= b.lo[0] && i + q < b.hi[0] ? w : T(0);
            s0[q] += comp == 0 ? x : T(0);
            s1[q] += comp == 1 ? x : T(0);
            s2[q] += comp == 2 ? x : T(0);
        }
    }
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        v0[q] += s0[q];
        v1[q] += s1[q];
        v2[q] += s2[q];
    }
}
template <typename T, int kV>
__device__ __forceinline__ bool in_sources(const CellArgs<T>& c, int i, int j, int kg) {
    return kg >= c.src_lo[2] && kg < c.src_hi[2] && j >= c.src_lo[1] && j < c.src_hi[1] && i + kV > c.src_lo[0] &&
           i < c.src_hi[0];
}

// DFT samples of components c0 .. c0 + 2 of a group (the values the update writes).
template <typename T, int kV>
__device__ __forceinline__ void put_samples(const CellArgs<T>& c, const StepArgs& a, int c0, int i, int j, int kg,
                                            const Group<T, kV>& v0, const Group<T, kV>& v1, const Group<T, kV>& v2) {
    if (!in_sample_plane(c, a, kg)) return;
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        if (!in_sample_rect(c, i + q, j)) continue;
        const long long o = sample_off(c, a, i + q, j, kg);
        if (c.smp[c0]) c.smp[c0][o] = v0[q];
        if (c.smp[c0 + 1]) c.smp[c0 + 1][o] = v1[q];
        if (c.smp[c0 + 2]) c.smp[c0 + 2][o] = v2[q];
    }
}

// Trapezoidal pole update of component a for the dispersive cells (bits of disp) of a group whose pole states start
// at offset bo; the arithmetic of ade_update.  kNP poles are held in registers between the two uses of their
// state; kNP = 0: any number, read twice.  kVec: the states of the group are one aligned vector.
template <typename T, int kV, int kNP, bool kVec>
__device__ __forceinline__ void ade_group(const Dom<T>& d, int a, long long bo, unsigned disp, Group<T, kV>& e,
                                          const Group<T, kV>& ie, const Group<T, kV>& scurl) {
    T* const base = d.ade + (long long)a * d.npole * 2 * d.bcell + bo;
    auto load = [&](const T* p) {
        if (kVec) return ld_group<T, kV>(p);
        Group<T, kV> g;
#pragma unroll
        for (int q = 0; q < kV; ++q) g[q] = disp >> q & 1 ? p[q] : T(0);
        return g;
    };
    auto store = [&](T* p, const Group<T, kV>& g) {
        if (kVec) {
            st_group(p, g);
            return;
        }
#pragma unroll
        for (int q = 0; q < kV; ++q)
            if (disp >> q & 1) p[q] = g[q];
    };
    const int np = kNP ? kNP : d.npole;
    Group<T, kV> P[kNP ? kNP : 1], Q[kNP ? kNP : 1], delta = scurl;
    if (kNP) {
#pragma unroll
        for (int p = 0; p < (kNP ? kNP : 1); ++p) {
            P[p] = load(base + (2 * p) * d.bcell);
            Q[p] = load(base + (2 * p + 1) * d.bcell);
        }
    }
#pragma unroll
    for (int p = 0; p < np; ++p) {
        if (!kNP) {
            P[0] = load(base + (2 * p) * d.bcell);
            Q[0] = load(base + (2 * p + 1) * d.bcell);
        }
        const int r = kNP ? p : 0;
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const T mp = fma_t(d.M00[p], P[r][q], d.M01[p] * Q[r][q]);
            delta[q] = delta[q] + fma_t(-T(2) * d.g0[p], e[q], P[r][q] - mp);
        }
    }
    Group<T, kV> es;
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        const T e1 = fma_t(ie[q] / fma_t(ie[q], d.G, T(1)), delta[q], e[q]);
        es[q] = e1 + e[q];
        if (disp >> q & 1) e[q] = e1;
    }
#pragma unroll
    for (int p = 0; p < np; ++p) {
        if (!kNP) {
            P[0] = load(base + (2 * p) * d.bcell);
            Q[0] = load(base + (2 * p + 1) * d.bcell);
        }
        const int r = kNP ? p : 0;
        Group<T, kV> P1 = P[r], Q1 = Q[r];
#pragma unroll
        for (int q = 0; q < kV; ++q)
            if (disp >> q & 1) {
                P1[q] = fma_t(d.g0[p], es[q], fma_t(d.M00[p], P[r][q], d.M01[p] * Q[r][q]));
                Q1[q] = fma_t(d.g1[p], es[q], fma_t(d.M10[p], P[r][q], d.M11[p] * Q[r][q]));
            }
        store(base + (2 * p) * d.bcell, P1);
        store(base + (2 * p + 1) * d.bcell, Q1);
    }
}
template <typename T, int kV>
__device__ __forceinline__ void ade_dispatch(const Dom<T>& d, int a, long long bo, bool vec, unsigned disp,
                                             Group<T, kV>& e, const Group<T, kV>& ie, const Group<T, kV>& scurl) {
    if (d.npole == 2) {
        if (vec) ade_group<T, kV, 2, true>(d, a, bo, disp, e, ie, scurl);
        else ade_group<T, kV, 2, false>(d, a, bo, disp, e, ie, scurl);
    } else if (vec) {
        ade_group<T, kV, 0, true>(d, a, bo, disp, e, ie, scurl);
    } else {
        ade_group<T, kV, 0, false>(d, a, bo, disp, e, ie, scurl);
    }
}

// kBack: the backward step of the reversible reconstruction (Sec. 3.2) for a lossless domain,
// E^n = (E^{n+1} - s^n) - S eps^-1 curl H^{n+1/2}, called with S negated (no CPML, no poles).
// kCurl: the first half of a tensor domain's E update (Sec. 2.3): the CPML-corrected curl of every
// non-PEC edge into c.cur (the memories advance as usual); launch_tensor_apply then applies S_t.
// block: this block's number among those of its region of plane k.
template <typename T, int kV, bool kEdge, bool kAniso, bool kPoles, bool kPer, bool kBack, bool kCurl>
__device__ __forceinline__ void e_cell_body(const CellArgs<T>& c, const Dom<T>* __restrict__ doms, T S,
                                            const StepArgs& a, unsigned block, int k) {
    using G = Group<T, kV>;
    const int nx = c.n[0], ny = c.n[1];
    const GroupAt at = group_at<T, kV, kEdge>(c, block);
    const int i = at.i, j = at.j;
    const int kg = k + c.kz0;   // global plane (CPML z profile, sources)
    const long long nxy = (long long)nx * ny;
    const long long id = (long long)k * nxy + (j * nx + i);
    const bool perx = kPer && c.per[0], pery = kPer && c.per[1];
    const T* Hx = c.F[3] + id;
    const T* Hy = c.F[4] + id;
    const T* Hz = c.F[5] + id;
    const G hx = ld_group<T, kV>(Hx), hy = ld_group<T, kV>(Hy), hz = ld_group<T, kV>(Hz);
    // -1 neighbours (wrapping on a periodic axis, else zero beyond a wall)
    G hz_ym{}, hx_ym{}, hx_zm{}, hy_zm{};
    if (j > 0 || pery) {
        const long long o = j > 0 ? -(long long)nx : nxy - nx;
        hz_ym = ld_group<T, kV>(Hz + o);
        hx_ym = ld_group<T, kV>(Hx + o);
    }
    if (k > 0) {
        hx_zm = ld_group<T, kV>(Hx - nxy);
        hy_zm = ld_group<T, kV>(Hy - nxy);
    }
    T hz_xm = T(0), hy_xm = T(0);
    if (i == 0 ? perx : !at.left) {
        const int o = i == 0 ? nx - 1 : -1;
        hz_xm = Hz[o];
        hy_xm = Hy[o];
    }
    G ex = ld_group<T, kV>(c.F[0] + id), ey = ld_group<T, kV>(c.F[1] + id), ez = ld_group<T, kV>(c.F[2] + id);
    const G iex = kCurl ? G{} : ld_group<T, kV>(c.ie[0] + id);
    const G iey = kAniso ? ld_group<T, kV>(c.ie[1] + id) : iex;
    const G iez = kAniso ? ld_group<T, kV>(c.ie[2] + id) : iex;
    GroupCpml<T, kV, kEdge> mem;
    if (!kBack) load_cpml(c, i, j, k, mem);
    const T zl = __shfl_up_sync(0xffffffffu, hz[kV - 1], 1), yl = __shfl_up_sync(0xffffffffu, hy[kV - 1], 1);
    if (!at.live) return;
    if (at.left) {
        hz_xm = zl;
        hy_xm = yl;
    }
    G yx1, yx2, yy1, yy2, yz1, yz2;
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        yx1[q] = hz[q] - hz_ym[q];                      // Ex: dHz/dy, dHy/dz
        yx2[q] = hy[q] - hy_zm[q];
        yy1[q] = hx[q] - hx_zm[q];                      // Ey: dHx/dz, dHz/dx
        yy2[q] = hz[q] - (q ? hz[q ? q - 1 : 0] : hz_xm);
        yz1[q] = hy[q] - (q ? hy[q ? q - 1 : 0] : hy_xm);   // Ez: dHy/dx, dHx/dy
        yz2[q] = hx[q] - hx_ym[q];
    }
    // PEC-held components: Ex on y = 0 and z = 0, Ey on x = 0 and z = 0, Ez on x = 0 and y = 0 (bit q: cell q)
    constexpr unsigned all = (1u << kV) - 1;
    const unsigned pi = i == 0 && !perx ? 1u : 0u, pjk = (j == 0 && !pery) || k == 0 ? all : 0u;
    const unsigned px = pjk, py = k == 0 ? all : pi, pz = j == 0 && !pery ? all : pi;
    if (kBack) {
        if (j < c.alo[1] || j >= c.ahi[1] || k < c.alo[2] || k >= c.ahi[2]) return;
        G sx{}, sy{}, sz{};
        if (in_sources<T, kV>(c, i, j, kg)) add_sources<T, kV>(c, a, 0, i, j, kg, sx, sy, sz);
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            if (i + q < c.alo[0] || i + q >= c.ahi[0]) continue;
            if (!(px >> q & 1)) ex[q] = fma_t(S * iex[q], (yx1[q] - yx2[q]), ex[q] - sx[q]);
            if (!(py >> q & 1)) ey[q] = fma_t(S * iey[q], (yy1[q] - yy2[q]), ey[q] - sy[q]);
            if (!(pz >> q & 1)) ez[q] = fma_t(S * iez[q], (yz1[q] - yz2[q]), ez[q] - sz[q]);
        }
        st_group(c.F[0] + id, ex);
        st_group(c.F[1] + id, ey);
        st_group(c.F[2] + id, ez);
        return;
    }
    apply_cpml(c, i, mem, yy2, yz1, yx1, yz2, yx2, yy1, px, py, pz);
    if (kCurl) {
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            if (!(px >> q & 1)) c.cur[0][id + q] = yx1[q] - yx2[q];
            if (!(py >> q & 1)) c.cur[1][id + q] = yy1[q] - yy2[q];
            if (!(pz >> q & 1)) c.cur[2][id + q] = yz1[q] - yz2[q];
        }
        return;
    }
    unsigned disp = 0;
    if (kPoles) {
        const Dom<T>& d = doms[c.dom];
        if (d.npole > 0 && j >= d.blo[1] && j < d.bhi[1] && k >= d.blo[2] && k < d.bhi[2]) {
#pragma unroll
            for (int q = 0; q < kV; ++q)
                if (i + q >= d.blo[0] && i + q < d.bhi[0] && d.mask[id + q]) disp |= 1u << q;
        }
        if (disp) {
            const long long bo = ade_off(d, i, j, k);
            // the group's states are one aligned vector where the box starts and ends on group boundaries
            const bool vec = kV > 1 && ((d.blo[0] | d.bhi[0]) & (kV - 1)) == 0;
            G sc;
#pragma unroll
            for (int q = 0; q < kV; ++q) sc[q] = mul_t(S, yx1[q] - yx2[q]);
            if (disp & ~px) ade_dispatch<T, kV>(d, 0, bo, vec, disp & ~px, ex, iex, sc);
#pragma unroll
            for (int q = 0; q < kV; ++q) sc[q] = mul_t(S, yy1[q] - yy2[q]);
            if (disp & ~py) ade_dispatch<T, kV>(d, 1, bo, vec, disp & ~py, ey, iey, sc);
#pragma unroll
            for (int q = 0; q < kV; ++q) sc[q] = mul_t(S, yz1[q] - yz2[q]);
            if (disp & ~pz) ade_dispatch<T, kV>(d, 2, bo, vec, disp & ~pz, ez, iez, sc);
        }
    }
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        if (kPoles && (disp >> q & 1)) continue;
        if (!(px >> q & 1)) ex[q] = fma_t(S * iex[q], (yx1[q] - yx2[q]), ex[q]);
        if (!(py >> q & 1)) ey[q] = fma_t(S * iey[q], (yy1[q] - yy2[q]), ey[q]);
        if (!(pz >> q & 1)) ez[q] = fma_t(S * iez[q], (yz1[q] - yz2[q]), ez[q]);
    }
    // (no source lies on a held node: fdtd_add_source refuses it; a held component keeps its value)
    if (in_sources<T, kV>(c, i, j, kg)) add_sources<T, kV>(c, a, 0, i, j, kg, ex, ey, ez);
    st_group(c.F[0] + id, ex);
    st_group(c.F[1] + id, ey);
    st_group(c.F[2] + id, ez);
    put_samples<T, kV>(c, a, 0, i, j, kg, ex, ey, ez);   // E^{n+1}
}

template <typename T, int kV, bool kAniso, bool kPoles, bool kPer, bool kBack = false, bool kCurl = false>
__global__ void __launch_bounds__(kCellThreads, cell_blocks<T, kV, kPoles>())
    k_e_cell(const __grid_constant__ CellArgs<T> c, const Dom<T>* __restrict__ doms, T S, const StepArgs a) {
    pdl_wait();
    if (blockIdx.x >= c.rows[0].nb)
        e_cell_body<T, edge_group(kV), true, kAniso, kPoles, kPer, kBack, kCurl>(c, doms, S, a, blockIdx.x - c.rows[0].nb, blockIdx.y);
    else
        e_cell_body<T, kV, false, kAniso, kPoles, kPer, kBack, kCurl>(c, doms, S, a, blockIdx.x, blockIdx.y);
}

// Domain of block b of a multi-domain launch: the last d with bbeg[d] <= b (bbeg: prefix sums of the
// domains' block counts); its argument block is copied into shared memory once per block.
template <typename T>
__device__ __forceinline__ void multi_cell(const CellArgs<T>* __restrict__ args, const int* __restrict__ bbeg, int ndom,
                                           int b, CellArgs<T>& sc, unsigned& block, int& k) {
    // every warp counts the prefix sums up to b with two loads a lane: one memory latency for up to 64 domains, and one more
    // for every 32nd of them that it takes first (64 steps of 512 / 2048 domains of 8^3 and 8192 of 4^3: 0.90 / 3.2 / 6.3 ms;
    // before plane_group 1.39 / 5.0 / 10.0, where counting through all of them took 1.48 / 7.1 / 35.9)
    const int lane = threadIdx.x & 31;
    int lo = 0, left = ndom;   // (bbeg[lo] <= b)
    while (left > 64) {
        const int step = (left + 31) >> 5;
        const int at = (__popc(__ballot_sync(0xffffffffu, lane * step < left && bbeg[lo + lane * step] <= b)) - 1) * step;
        lo += at;
        left = min(step, left - at);
    }
    const unsigned low = __ballot_sync(0xffffffffu, lane < left && bbeg[lo + lane] <= b);
    const unsigned high = __ballot_sync(0xffffffffu, lane + 32 < left && bbeg[lo + lane + 32] <= b);
    lo += __popc(low) + __popc(high) - 1;
    const int* src = (const int*)(args + lo);
    int* dst = (int*)&sc;
    for (int w = threadIdx.x; w < (int)(sizeof(CellArgs<T>) / sizeof(int)); w += kCellThreads) dst[w] = src[w];
    __syncthreads();
    const unsigned local = b - bbeg[lo], per = sc.rows[0].nb + sc.rows[1].nb;
    k = local / per;
    block = local - k * per;
}

// Every domain of a batch in one launch (per-cell launch mode with several domains): the same body as
// k_e_cell, the domain's operands read from its argument block.
template <typename T, int kV, bool kAniso, bool kPoles, bool kPer>
__global__ void __launch_bounds__(kCellThreads, cell_blocks<T, kV, kPoles>())
    k_e_cells(const CellArgs<T>* __restrict__ args, const int* __restrict__ bbeg, int ndom,
              const Dom<T>* __restrict__ doms, T S, const StepArgs a) {
    __shared__ CellArgs<T> sc;
    unsigned block;
    int k;
    multi_cell(args, bbeg, ndom, blockIdx.x, sc, block, k);
    pdl_wait();
    if (block >= sc.rows[0].nb)
        e_cell_body<T, edge_group(kV), true, kAniso, kPoles, kPer, false, false>(sc, doms, S, a, block - sc.rows[0].nb, k);
    else
        e_cell_body<T, kV, false, kAniso, kPoles, kPer, false, false>(sc, doms, S, a, block, k);
}

// kBack: backward H step, H^{n+1/2} = (H^{n+3/2} - m^n) + S curl E^{n+1}, called with S negated.  Returns (kEnergy) the
// group's part of the discrete energy W_{n+1} = 1/2 sum eps |E|^2 + 1/2 sum H^{n+1/2} . H^{n+3/2}.
template <typename T, int kV, bool kEdge, bool kPer, bool kBack, bool kEnergy>
__device__ __forceinline__ double h_cell_body(const CellArgs<T>& c, T S, const StepArgs& a, unsigned block, int k) {
    using G = Group<T, kV>;
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    const GroupAt at = group_at<T, kV, kEdge>(c, block);
    const int i = at.i, j = at.j;
    const int kg = k + c.kz0;   // global plane (CPML z profile, sources)
    const long long nxy = (long long)nx * ny;
    const long long id = (long long)k * nxy + (j * nx + i);
    const bool perx = kPer && c.per[0], pery = kPer && c.per[1];
    const T* Ex = c.F[0] + id;
    const T* Ey = c.F[1] + id;
    const T* Ez = c.F[2] + id;
    const G ex = ld_group<T, kV>(Ex), ey = ld_group<T, kV>(Ey), ez = ld_group<T, kV>(Ez);
    // +1 neighbours (wrapping on a periodic axis, else zero: the node does not exist)
    G ez_yp{}, ex_yp{}, ey_zp{}, ex_zp{};
    if (j + 1 < ny || pery) {
        const long long o = j + 1 < ny ? (long long)nx : nx - nxy;
        ez_yp = ld_group<T, kV>(Ez + o);
        ex_yp = ld_group<T, kV>(Ex + o);
    }
    if (k + 1 < nz) {
        ey_zp = ld_group<T, kV>(Ey + nxy);
        ex_zp = ld_group<T, kV>(Ex + nxy);
    }
    const bool last = i + kV >= nx;   // the group ends its row
    T ez_xp = T(0), ey_xp = T(0);
    if (last ? perx : !at.right) {
        const int o = last ? kV - nx : kV;
        ez_xp = Ez[o];
        ey_xp = Ey[o];
    }
    G hx = ld_group<T, kV>(c.F[3] + id), hy = ld_group<T, kV>(c.F[4] + id), hz = ld_group<T, kV>(c.F[5] + id);
    GroupCpml<T, kV, kEdge> mem;
    if (!kBack) load_cpml(c, i, j, k, mem);
    const T zr = __shfl_down_sync(0xffffffffu, ez[0], 1), yr = __shfl_down_sync(0xffffffffu, ey[0], 1);
    if (!at.live) return 0.0;
    if (at.right) {
        ez_xp = zr;
        ey_xp = yr;
    }
    const G ox = hx, oy = hy, oz = hz;   // H^{n+1/2}
    G yx1, yx2, yy1, yy2, yz1, yz2;
#pragma unroll
    for (int q = 0; q < kV; ++q) {
        constexpr int e = kV - 1;
        yx1[q] = ez_yp[q] - ez[q];                                  // Hx: dEz/dy, dEy/dz
        yx2[q] = ey_zp[q] - ey[q];
        yy1[q] = ex_zp[q] - ex[q];                                  // Hy: dEx/dz, dEz/dx
        yy2[q] = (q < e ? ez[q < e ? q + 1 : 0] : ez_xp) - ez[q];
        yz1[q] = (q < e ? ey[q < e ? q + 1 : 0] : ey_xp) - ey[q];   // Hz: dEy/dx, dEx/dy
        yz2[q] = ex_yp[q] - ex[q];
    }
    if (kBack) {
        if (j < c.alo[1] || j >= c.ahi[1] || k < c.alo[2] || k >= c.ahi[2]) return 0.0;
        G mx{}, my{}, mz{};
        if (in_sources<T, kV>(c, i, j, kg)) add_sources<T, kV>(c, a, 3, i, j, kg, mx, my, mz);
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            if (i + q < c.alo[0] || i + q >= c.ahi[0]) continue;
            hx[q] = fma_t(-S, (yx1[q] - yx2[q]), hx[q] - mx[q]);
            hy[q] = fma_t(-S, (yy1[q] - yy2[q]), hy[q] - my[q]);
            hz[q] = fma_t(-S, (yz1[q] - yz2[q]), hz[q] - mz[q]);
        }
    } else {
        apply_cpml(c, i, mem, yy2, yz1, yx1, yz2, yx2, yy1, 0u, 0u, 0u);
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            hx[q] = fma_t(-S, (yx1[q] - yx2[q]), hx[q]);
            hy[q] = fma_t(-S, (yy1[q] - yy2[q]), hy[q]);
            hz[q] = fma_t(-S, (yz1[q] - yz2[q]), hz[q]);
        }
        if (in_sources<T, kV>(c, i, j, kg)) add_sources<T, kV>(c, a, 3, i, j, kg, hx, hy, hz);
    }
    st_group(c.F[3] + id, hx);
    st_group(c.F[4] + id, hy);
    st_group(c.F[5] + id, hz);
    if (!kBack) put_samples<T, kV>(c, a, 3, i, j, kg, hx, hy, hz);   // H^{n+3/2}
    double w = 0.0;
    if (kEnergy) {
        const bool iso = c.ie[1] == c.ie[0] && c.ie[2] == c.ie[0];
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            w += (double)ox[q] * hx[q] + (double)oy[q] * hy[q] + (double)oz[q] * hz[q];
            // (an isotropic cell's three terms share their FP64 division)
            const double x = (double)ex[q] * ex[q], y = (double)ey[q] * ey[q], z = (double)ez[q] * ez[q];
            if (iso) w += (x + y + z) / (double)c.ie[0][id + q];
            else w += x / (double)c.ie[0][id + q] + y / (double)c.ie[1][id + q] + z / (double)c.ie[2][id + q];
        }
    }
    return 0.5 * w;
}

// Adds the energy parts of a block's threads to the domain's record of this step: one atomic a block.
template <typename T>
__device__ __forceinline__ void add_energy(const CellArgs<T>& c, const StepArgs& a, double w) {
    __shared__ double part[kCellThreads / 32];
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int q = 1; q < kCellThreads / 32; ++q) w += part[q];
    const int step = *a.d_base + a.offset;
    if (c.energy && step < c.energy_cap) atomicAdd(c.energy + step, w);
}

template <typename T, int kV, bool kPer, bool kBack = false, bool kEnergy = false>
__global__ void __launch_bounds__(kCellThreads, cell_blocks<T, kV>())
    k_h_cell(const __grid_constant__ CellArgs<T> c, T S, const StepArgs a) {
    pdl_wait();
    // planes last to first (the E kernels run first to last): the planes the half-step before has just touched are
    // still in L2
    const int k = (int)(gridDim.y - 1 - blockIdx.y);
    double w;
    if (blockIdx.x >= c.rows[0].nb)
        w = h_cell_body<T, edge_group(kV), true, kPer, kBack, kEnergy>(c, S, a, blockIdx.x - c.rows[0].nb, k);
    else
        w = h_cell_body<T, kV, false, kPer, kBack, kEnergy>(c, S, a, blockIdx.x, k);
    if (kEnergy) add_energy(c, a, w);
}

template <typename T, int kV, bool kPer, bool kEnergy>
__global__ void __launch_bounds__(kCellThreads, cell_blocks<T, kV>())
    k_h_cells(const CellArgs<T>* __restrict__ args, const int* __restrict__ bbeg, int ndom, T S, const StepArgs a) {
    __shared__ CellArgs<T> sc;
    unsigned block;
    int k;
    multi_cell(args, bbeg, ndom, gridDim.x - 1 - blockIdx.x, sc, block, k);   // last to first, as k_h_cell
    pdl_wait();
    double w;
    if (block >= sc.rows[0].nb)
        w = h_cell_body<T, edge_group(kV), true, kPer, false, kEnergy>(sc, S, a, block - sc.rows[0].nb, k);
    else
        w = h_cell_body<T, kV, false, kPer, false, kEnergy>(sc, S, a, block, k);
    if (kEnergy) add_energy(sc, a, w);
}

// Cells per thread along x: the longest group that divides the rows and to which every array the update reads or
// writes by groups is aligned (fields and CPML memories along y and z are whole allocations or whole planes of
// them; eps^-1 is the caller's).  FP64: one cell (see cell_blocks).
template <typename T>
int cell_group(const CellArgs<T>& c) {
    int v = sizeof(T) == 4 ? 4 : 1;
    auto fits = [&](const void* p) {
        while (v > 1 && (uintptr_t)p % (v * sizeof(T))) v /= 2;
    };
    while (v > 1 && c.n[0] % v) v /= 2;
    for (const T* p : c.F) fits(p);
    for (const T* p : c.ie) fits(p);
    for (int q = 1; q < 3; ++q) {   // the memories of the derivatives along y and z
        fits(c.psi[(q + 1) % 3][1]);
        fits(c.psi[(q + 2) % 3][0]);
    }
    return v;
}

// The two regions of a plane (see group_at) for groups of v cells.
template <typename T>
void set_groups(CellArgs<T>& c, int v) {
    const int nx = c.n[0], e = edge_group(v);
    int lo = c.ns[0] ? (c.dlo[0] + v - 1) / v * v : 0, hi = c.ns[0] ? (c.dhi[0] + v - 1) / v * v : 0;
    // no group without slab cells, or a plane that fits one block as a whole (its slab columns apart would take a second one:
    // a step of 2048 planes of 16 x 16 with slabs 9.5 us against 15.0)
    if (lo + hi >= nx || (lo + hi > 0 && (long long)(nx / e) * c.n[1] <= kCellThreads)) {
        lo = nx;
        hi = 0;
    }
    c.xlo = lo;
    c.xin = nx - lo - hi;
    c.rows[0] = make_rows((unsigned)(c.xin / v), c.n[1]);
    c.rows[1] = make_rows((unsigned)((lo + hi) / e), c.n[1]);
    // the memories along x by groups: their rows divide into groups (then the first slab index of every group does,
    // as e divides nx), and so do their addresses
    c.xvec = c.ns[0] % e == 0 && (uintptr_t)c.psi[1][1] % (e * sizeof(T)) == 0 &&
             (uintptr_t)c.psi[2][0] % (e * sizeof(T)) == 0;
}

// grid: blocks of a plane, z planes
template <typename T>
inline dim3 cell_grid(const CellArgs<T>& c) {
    return dim3(c.rows[0].nb + c.rows[1].nb, (unsigned)c.n[2]);
}

template <typename T>
void launch_e_cell(const Launch& L, const CellArgs<T>& c0, const Dom<T>* doms, T S, const StepArgs& a, int aniso,
                   int poles) {
    CellArgs<T> c = c0;
    const int v = plane_group((long long)c.n[0] * c.n[1], cell_group(c));
    set_groups(c, v);
    with_group<T>(v, [&](auto V) {
        with_bool(aniso, [&](auto A) {
            with_bool(poles, [&](auto P) {
                with_bool(c.per[0] || c.per[1], [&](auto R) {
                    launch_k(L, k_e_cell<T, V(), A(), P(), R()>, cell_grid(c), dim3(kCellThreads), c, doms, S, a);
                });
            });
        });
    });
    ++*L.counter;
}

template <typename T>
void launch_h_cell(const Launch& L, const CellArgs<T>& c0, T S, const StepArgs& a, int energy) {
    CellArgs<T> c = c0;
    const int v = plane_group((long long)c.n[0] * c.n[1], cell_group(c));
    set_groups(c, v);
    with_group<T>(v, [&](auto V) {
        with_bool(c.per[0] || c.per[1], [&](auto R) {
            with_bool(energy, [&](auto E) {
                launch_k(L, k_h_cell<T, V(), R(), false, E()>, cell_grid(c), dim3(kCellThreads), c, S, a);
            });
        });
    });
    ++*L.counter;
}

template <typename T>
int prepare_cells(CellArgs<T>* args, int* bbeg, int ndom, int v) {
    long long cells = 0, planes = 0;
    for (int d = 0; d < ndom; ++d) {
        v = std::min(v, cell_group(args[d]));
        cells += (long long)args[d].n[0] * args[d].n[1] * args[d].n[2];
        planes += args[d].n[2];
    }
    v = plane_group(cells / planes, v);   // one length for the batch: that of its mean plane
    bbeg[0] = 0;
    for (int d = 0; d < ndom; ++d) {
        set_groups(args[d], v);
        const dim3 g = cell_grid(args[d]);
        bbeg[d + 1] = bbeg[d] + (int)(g.x * g.y);
    }
    return v;
}

template <typename T>
void launch_e_cells(const Launch& L, const CellArgs<T>* args, const int* bbeg, int ndom, int nblocks, int v,
                    const Dom<T>* doms, T S, const StepArgs& a, int aniso, int poles, int per) {
    with_group<T>(v, [&](auto V) {
        with_bool(aniso, [&](auto A) {
            with_bool(poles, [&](auto P) {
                with_bool(per, [&](auto R) {
                    launch_k(L, k_e_cells<T, V(), A(), P(), R()>, dim3(nblocks), dim3(kCellThreads), args, bbeg, ndom, doms, S, a);
                });
            });
        });
    });
    ++*L.counter;
}

template <typename T>
void launch_h_cells(const Launch& L, const CellArgs<T>* args, const int* bbeg, int ndom, int nblocks, int v, T S,
                    const StepArgs& a, int per, int energy) {
    with_group<T>(v, [&](auto V) {
        with_bool(per, [&](auto R) {
            with_bool(energy, [&](auto E) {
                launch_k(L, k_h_cells<T, V(), R(), E()>, dim3(nblocks), dim3(kCellThreads), args, bbeg, ndom, S, a);
            });
        });
    });
    ++*L.counter;
}

template <typename T>
void launch_e_curl(const Launch& L, const CellArgs<T>& c0) {
    CellArgs<T> c = c0;
    const int v = plane_group((long long)c.n[0] * c.n[1], cell_group(c));
    set_groups(c, v);
    with_group<T>(v, [&](auto V) {
        with_bool(c.per[0] || c.per[1], [&](auto R) {
            k_e_cell<T, V(), false, false, R(), false, true>
                <<<cell_grid(c), kCellThreads, 0, L.stream>>>(c, nullptr, T(0), StepArgs{});
        });
    });
    ++*L.counter;
}

template <typename T>
void launch_back_h(const Launch& L, const CellArgs<T>& c0, T S, const StepArgs& a) {
    CellArgs<T> c = c0;
    const int v = plane_group((long long)c.n[0] * c.n[1], cell_group(c));
    set_groups(c, v);
    with_group<T>(v, [&](auto V) {
        with_bool(c.per[0] || c.per[1], [&](auto R) {
            k_h_cell<T, V(), R(), true><<<cell_grid(c), kCellThreads, 0, L.stream>>>(c, -S, a);
        });
    });
    ++*L.counter;
}

template <typename T>
void launch_back_e(const Launch& L, const CellArgs<T>& c0, T S, const StepArgs& a, int aniso) {
    CellArgs<T> c = c0;
    const int v = plane_group((long long)c.n[0] * c.n[1], cell_group(c));
    set_groups(c, v);
    with_group<T>(v, [&](auto V) {
        with_bool(aniso, [&](auto A) {
            with_bool(c.per[0] || c.per[1], [&](auto R) {
                k_e_cell<T, V(), A(), false, R(), true><<<cell_grid(c), kCellThreads, 0, L.stream>>>(c, nullptr, -S, a);
            });
        });
    });
    ++*L.counter;
}

// Backward step of a lossless domain: the H kernel first (it reads E^{n+1}), then the E kernel.
template <typename T>
void launch_back_cell(const Launch& L, const CellArgs<T>& ce, const CellArgs<T>& ch, T S, const StepArgs& a,
                      int aniso) {
    launch_back_h<T>(L, ch, S, a);
    launch_back_e<T>(L, ce, S, a, aniso);
}

// Interface planes <-> record slot (see IfaceArgs): blockIdx.y picks the plane, threads run over
// its three components x cells.
template <typename T>
__global__ void __launch_bounds__(256) k_iface(const int n0, const int n1, const int n2, const IfaceArgs ia,
                                               T* __restrict__ rec, const int* __restrict__ d_base, int bias, int kinds,
                                               int to_rec, T* Ex, T* Ey, T* Ez, T* Hx, T* Hy, T* Hz) {
    if (blockIdx.y >= (unsigned)ia.np) return;
    const IfacePlane pl = ia.p[blockIdx.y];
    if (!((kinds >> pl.kind) & 1)) return;   // kind 0 = H (bit 0), 1 = E (bit 1)
    const long long s = (long long)(d_base ? *d_base : 0) + bias - ia.t0;
    if (s < 0 || s > ia.cap) return;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * pl.cells) return;
    const int comp = (int)(t / pl.cells);
    const long long cell = t - (long long)comp * pl.cells;
    // plane cell -> (i, j, k): the two other axes in increasing order, the first one fastest
    int c[3];
    const int nn[3] = {n0, n1, n2};
    const int a0 = pl.q == 0 ? 1 : 0, a1 = pl.q == 2 ? 1 : 2;
    c[pl.q] = pl.x;
    c[a0] = (int)(cell % nn[a0]);
    c[a1] = (int)(cell / nn[a0]);
    const long long id = ((long long)c[2] * n1 + c[1]) * n0 + c[0];
    T* fields[6] = {Ex, Ey, Ez, Hx, Hy, Hz};
    T* f = fields[(pl.kind == 0 ? 3 : 0) + comp];
    T* r = rec + s * ia.slot + pl.off + t;
    if (to_rec)
        *r = f[id];
    else
        f[id] = *r;
}

template <typename T>
void launch_iface(const Launch& L, T* const* F, const int* n, const IfaceArgs& ia, T* rec, const int* d_base, int bias,
                  int kinds, int to_rec) {
    if (ia.np <= 0) return;
    long long most = 0;
    for (int q = 0; q < ia.np; ++q) most = most > 3 * ia.p[q].cells ? most : 3 * ia.p[q].cells;
    const dim3 g((unsigned)((most + 255) / 256), (unsigned)ia.np);
    k_iface<T><<<g, 256, 0, L.stream>>>(n[0], n[1], n[2], ia, rec, d_base, bias, kinds, to_rec, F[0], F[1], F[2], F[3],
                                         F[4], F[5]);
    ++*L.counter;
}

__global__ void k_advance(int* d_step, int delta) { *d_step += delta; }

// ---- host launchers --------------------------------------------------------------------------
template <typename T>
void launch_e_update(const Launch& L, const Dom<T>* doms, const Tile* tiles, int ntiles, T S, const StepArgs& a,
                     int general, int aniso) {
    if (ntiles <= 0) return;
    const dim3 b(kTileX, kTileY);
    if (general)
        k_e_update<T, true, true><<<ntiles, b, 0, L.stream>>>(doms, tiles, S, a);
    else
        (aniso ? k_e_update<T, false, true> : k_e_update<T, false, false>)<<<ntiles, b, 0, L.stream>>>(doms, tiles, S,
                                                                                                     a);
    ++*L.counter;
}

template <typename T>
void launch_h_update(const Launch& L, const Dom<T>* doms, const Tile* tiles, int ntiles, T S, const StepArgs& a,
                     int general, int energy, unsigned advance) {
    if (ntiles <= 0) return;
    const dim3 b(kTileX, kTileY);
    if (general)
        (energy ? k_h_update<T, true, true> : k_h_update<T, true, false>)<<<ntiles, b, 0, L.stream>>>(doms, tiles, S, a,
                                                                                                    advance);
    else
        (energy ? k_h_update<T, false, true> : k_h_update<T, false, false>)<<<ntiles, b, 0, L.stream>>>(
            doms, tiles, S, a, advance);
    ++*L.counter;
}

template <typename T>
void launch_dft(const Launch& L, const Dom<T>* doms, const Mon* mons, const DftItem* items, int nitems, int kind,
                const int* d_base, int offset) {
    if (nitems <= 0) return;
    k_dft<T><<<nitems, dim3(kTileX, kTileY), 0, L.stream>>>(doms, mons, items, kind, d_base, offset);
    ++*L.counter;
}

template <typename T>
void launch_dft_ring(const Launch& L, const Mon* mons, const DftItem* items, int nitems, const int* d_base, int t0,
                     int cnt) {
    if (nitems <= 0 || cnt <= t0) return;
    // one grid row per component slot (6 at most; rows past a monitor's components return at once)
    k_dft_ring<T><<<dim3(nitems, 6), dim3(kTileX, kTileY), 0, L.stream>>>(mons, items, d_base, t0, cnt);
    ++*L.counter;
}

void launch_copy_int(const Launch& L, const int* src, int* dst) {
    k_copy_int<<<1, 1, 0, L.stream>>>(src, dst);
    ++*L.counter;
}

void launch_set_int(const Launch& L, int* dst, int v) {
    k_set_int<<<1, 1, 0, L.stream>>>(dst, v);
    ++*L.counter;
}

void launch_advance(const Launch& L, int* d_step, int delta) {
    k_advance<<<1, 1, 0, L.stream>>>(d_step, delta);
    ++*L.counter;
}

#define GBFDTD_INST(T)                                                                                           \
    template void launch_e_update<T>(const Launch&, const Dom<T>*, const Tile*, int, T, const StepArgs&, int, int); \
    template void launch_h_update<T>(const Launch&, const Dom<T>*, const Tile*, int, T, const StepArgs&, int, int,  \
                                     unsigned);
GBFDTD_INST(float)
GBFDTD_INST(double)
#undef GBFDTD_INST
template void launch_dft<float>(const Launch&, const Dom<float>*, const Mon*, const DftItem*, int, int, const int*,
                                int);
template void launch_dft<double>(const Launch&, const Dom<double>*, const Mon*, const DftItem*, int, int, const int*,
                                 int);
template void launch_dft_ring<float>(const Launch&, const Mon*, const DftItem*, int, const int*, int, int);
template void launch_dft_ring<double>(const Launch&, const Mon*, const DftItem*, int, const int*, int, int);
template void launch_e_cell<float>(const Launch&, const CellArgs<float>&, const Dom<float>*, float, const StepArgs&,
                                   int, int);
template void launch_e_cell<double>(const Launch&, const CellArgs<double>&, const Dom<double>*, double,
                                    const StepArgs&, int, int);
template void launch_back_cell<float>(const Launch&, const CellArgs<float>&, const CellArgs<float>&, float,
                                      const StepArgs&, int);
template void launch_back_cell<double>(const Launch&, const CellArgs<double>&, const CellArgs<double>&, double,
                                       const StepArgs&, int);
template void launch_back_h<float>(const Launch&, const CellArgs<float>&, float, const StepArgs&);
template void launch_back_h<double>(const Launch&, const CellArgs<double>&, double, const StepArgs&);
template void launch_back_e<float>(const Launch&, const CellArgs<float>&, float, const StepArgs&, int);
template void launch_back_e<double>(const Launch&, const CellArgs<double>&, double, const StepArgs&, int);
template void launch_iface<float>(const Launch&, float* const*, const int*, const IfaceArgs&, float*, const int*, int,
                                  int, int);
template void launch_iface<double>(const Launch&, double* const*, const int*, const IfaceArgs&, double*, const int*,
                                   int, int, int);
template int prepare_cells<float>(CellArgs<float>*, int*, int, int);
template int prepare_cells<double>(CellArgs<double>*, int*, int, int);
template void launch_e_cells<float>(const Launch&, const CellArgs<float>*, const int*, int, int, int,
                                    const Dom<float>*, float, const StepArgs&, int, int, int);
template void launch_e_cells<double>(const Launch&, const CellArgs<double>*, const int*, int, int, int,
                                     const Dom<double>*, double, const StepArgs&, int, int, int);
template void launch_h_cells<float>(const Launch&, const CellArgs<float>*, const int*, int, int, int, float,
                                    const StepArgs&, int, int);
template void launch_h_cells<double>(const Launch&, const CellArgs<double>*, const int*, int, int, int, double,
                                     const StepArgs&, int, int);
template void launch_e_curl<float>(const Launch&, const CellArgs<float>&);
template void launch_e_curl<double>(const Launch&, const CellArgs<double>&);
template void launch_h_cell<float>(const Launch&, const CellArgs<float>&, float, const StepArgs&, int);
template void launch_h_cell<double>(const Launch&, const CellArgs<double>&, double, const StepArgs&, int);

}  // namespace gbfdtd
