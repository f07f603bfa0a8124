// Auxiliary kernels: the CPML tensor admission rule (Sec. 2.3), the bounding box of the pole
// mask, a NaN/Inf scan, and the BF16 snapshot codec with one scale per slab (Sec. 3.2).
#include <cuda_bf16.h>

#include <cooperative_groups.h>

#include <algorithm>

#include "fdtd_internal.cuh"

namespace gbfdtd {

// Sec. 2.3: inside an absorbing face a tensor is admitted only if the face normal is a principal
// axis with a non-intermediate eigenvalue.  For a diagonal tensor the normal of a q-face is a
// principal axis; reject a cell of a q-slab whose eps_qq lies strictly between the other two
// (the same order test on 1/eps).
template <typename T>
__global__ void k_admission(const Dom<T>* __restrict__ dd, unsigned long long* bad) {
    const Dom<T>& d = *dd;
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= d.ncell) return;
    const int i = (int)(t % d.n[0]);
    const int j = (int)((t / d.n[0]) % d.n[1]);
    const int k = (int)(t / ((long long)d.n[0] * d.n[1]));
    const int c[3] = {i, j, k};
    const T v[3] = {d.ie[0][t], d.ie[1][t], d.ie[2][t]};
    for (int q = 0; q < 3; ++q) {
        if (d.ns[q] == 0 || slab_of(c[q], d.dlo[q], d.dhi[q], d.n[q]) < 0) continue;
        const T a = v[(q + 1) % 3], b = v[(q + 2) % 3], x = v[q];
        const T lo = a < b ? a : b, hi = a < b ? b : a;
        if (x > lo && x < hi) {
            atomicAdd(bad, 1ull);
            return;
        }
    }
}

__global__ void k_mask_box(const uint8_t* __restrict__ mask, int nx, int ny, int nz, int* box) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)nx * ny * nz) return;
    if (!mask[t]) return;
    const int i = (int)(t % nx), j = (int)((t / nx) % ny), k = (int)(t / ((long long)nx * ny));
    atomicMin(box + 0, i);
    atomicMin(box + 1, j);
    atomicMin(box + 2, k);
    atomicMax(box + 3, i + 1);
    atomicMax(box + 4, j + 1);
    atomicMax(box + 5, k + 1);
}

template <typename T>
__global__ void k_nonfinite(const T* __restrict__ p, long long n, unsigned long long* bad) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const T v = p[t];
        if (!(v == v) || v - v != T(0)) {  // NaN fails v == v; +-Inf gives Inf - Inf = NaN
            atomicAdd(bad, 1ull);
            return;
        }
    }
}

// BF16 snapshot codec, one FP32 scale per slab (outermost index): s = max |x| over the slab, q = bf16_rn(x / s), x' =
// float(q) * s.  One launch codes every slab of every state part: what bounded the form with three launches per
// part was their number (a 128^3 two-pole state has 30 parts: 60 launches and 30 memsets a save, 3.5 us each; the
// layer gradient of the benchmarks spent 22 of 51 ms in them and 14 in the gaps between).  A cluster of gridDim.x
// blocks takes a slab: it reads it for the maximum, exchanges the blocks' maxima through distributed shared memory,
// and reads it again (from L1 / L2) to quantise.  NaN is ignored by fmaxf, as in a sequential max.
constexpr int kCodecThreads = 512;

// Slab first + blockIdx.y -> its part and index in it (seg[q].slab0: the slabs of the parts before q).
__device__ __forceinline__ const CodecSeg& codec_seg(const CodecSeg* __restrict__ segs, int nseg, int first,
                                                     long long& slab) {
    int lo = 0, hi = nseg - 1;
    const int b = first + blockIdx.y;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (segs[mid].slab0 <= b) lo = mid;
        else hi = mid - 1;
    }
    slab = b - segs[lo].slab0;
    return segs[lo];
}

// Calls f(t, kN) for the values [begin, end) of a slab whose arrays start at multiples of 4 values if vec: kN = 4
// values at t, else 1.
template <typename F>
__device__ __forceinline__ void codec_range(long long begin, long long end, bool vec, F f) {
    if (vec) {
        for (long long t = begin + 4ll * threadIdx.x; t < end; t += 4ll * blockDim.x) {
            if (t + 4 <= end) {
                f(t, std::integral_constant<int, 4>{});
            } else {
                for (long long u = t; u < end; ++u) f(u, std::integral_constant<int, 1>{});
            }
        }
    } else {
        for (long long t = begin + threadIdx.x; t < end; t += blockDim.x) f(t, std::integral_constant<int, 1>{});
    }
}
// This block's part of a slab of n values: whole groups of four.
__device__ __forceinline__ void codec_share(long long n, long long& begin, long long& end) {
    const long long q = ((n + 4ll * gridDim.x - 1) / (4ll * gridDim.x)) * 4;
    begin = min(n, q * blockIdx.x);
    end = min(n, begin + q);
}

template <typename T>
__global__ void __launch_bounds__(kCodecThreads) k_bf16_encode(const CodecSeg* __restrict__ segs, int nseg,
                                                               int first, char* __restrict__ slot) {
    namespace cg = cooperative_groups;
    long long slab;
    const CodecSeg sg = codec_seg(segs, nseg, first, slab);
    const T* src = (const T*)sg.state + slab * sg.plane;
    __nv_bfloat16* dst = (__nv_bfloat16*)(slot + sg.codes) + slab * sg.plane;
    float* scale = (float*)(slot + sg.scales) + slab;
    const bool vec = sg.plane % 4 == 0 && ((uintptr_t)src % (4 * sizeof(T))) == 0 && ((uintptr_t)dst % 8) == 0;
    long long begin, end;
    codec_share(sg.plane, begin, end);
    float m = 0.f;
    codec_range(begin, end, vec, [&](long long t, auto n) {
        const Group<T, n()> g = ld_group<T, n()>(src + t);
#pragma unroll
        for (int q = 0; q < n(); ++q) m = fmaxf(m, fabsf((float)g[q]));
    });
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ float red[kCodecThreads / 32];
    __shared__ float mine;
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kCodecThreads / 32; ++w) m = fmaxf(m, red[w]);
        mine = m;
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    float s = 0.f;
    for (unsigned r = 0; r < cl.num_blocks(); ++r) s = fmaxf(s, *cl.map_shared_rank(&mine, r));
    cl.sync();   // no block leaves while another may still read its maximum
    if (blockIdx.x == 0 && threadIdx.x == 0) *scale = s;
    // divide (not multiply by 1/s): a slab whose max is an FP32 denormal has 1/s = inf, and 0 * inf would store NaN;
    // x / s stays within [-1, 1]
    codec_range(begin, end, vec, [&](long long t, auto n) {
        const Group<T, n()> g = ld_group<T, n()>(src + t);
        Group<__nv_bfloat16, n()> c;
#pragma unroll
        for (int q = 0; q < n(); ++q) c[q] = __float2bfloat16_rn(s > 0.f ? (float)g[q] / s : 0.f);
        st_group(dst + t, c);
    });
}

template <typename T>
__global__ void __launch_bounds__(kCodecThreads) k_bf16_decode(const CodecSeg* __restrict__ segs, int nseg,
                                                               int first, const char* __restrict__ slot) {
    long long slab;
    const CodecSeg sg = codec_seg(segs, nseg, first, slab);
    T* dst = (T*)sg.state + slab * sg.plane;
    const __nv_bfloat16* src = (const __nv_bfloat16*)(slot + sg.codes) + slab * sg.plane;
    const float s = ((const float*)(slot + sg.scales))[slab];
    const bool vec = sg.plane % 4 == 0 && ((uintptr_t)dst % (4 * sizeof(T))) == 0 && ((uintptr_t)src % 8) == 0;
    long long begin, end;
    codec_share(sg.plane, begin, end);
    codec_range(begin, end, vec, [&](long long t, auto n) {
        const Group<__nv_bfloat16, n()> c = ld_group<__nv_bfloat16, n()>(src + t);
        Group<T, n()> g;
#pragma unroll
        for (int q = 0; q < n(); ++q) g[q] = (T)(__bfloat162float(c[q]) * s);
        st_group(dst + t, g);
    });
}

// Net Poynting flux along +z through the H plane of a two-plane monitor (Sec. 2.4), one block
// per frequency: P = 1/2 Re sum [ (Ex(k) + Ex(k+1))/2 conj(Hy(k)) - (Ey(k) + Ey(k+1))/2 conj(Hx(k)) ]
// over the monitor's x-y cells.  sEx..sHy: accumulator slots of the four components.
__global__ void __launch_bounds__(256) k_flux(const Mon* __restrict__ mon, int sEx, int sEy, int sHx, int sHy,
                                              double* __restrict__ out) {
    const Mon& m = *mon;
    const int f = blockIdx.x;
    const long long plane = (long long)m.bx * m.by;
    const double2* ex = m.acc + ((long long)sEx * m.nf + f) * m.ncell;
    const double2* ey = m.acc + ((long long)sEy * m.nf + f) * m.ncell;
    const double2* hx = m.acc + ((long long)sHx * m.nf + f) * m.ncell;
    const double2* hy = m.acc + ((long long)sHy * m.nf + f) * m.ncell;
    double sum = 0.0;
    for (long long c = threadIdx.x; c < plane; c += blockDim.x) {
        const double2 a0 = ex[c], a1 = ex[c + plane], b0 = ey[c], b1 = ey[c + plane];
        const double2 gx = hx[c], gy = hy[c];
        const double exr = 0.5 * (a0.x + a1.x), exi = 0.5 * (a0.y + a1.y);
        const double eyr = 0.5 * (b0.x + b1.x), eyi = 0.5 * (b0.y + b1.y);
        // Re(E conj(H)) = Er Hr + Ei Hi
        sum += 0.5 * ((exr * gy.x + exi * gy.y) - (eyr * gx.x + eyi * gx.y));
    }
    __shared__ double red[256];
    red[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[f] = red[0];
}

void launch_flux(const Launch& L, const Mon* mon, int nf, const int* slots, double* out) {
    if (nf <= 0) return;
    k_flux<<<nf, 256, 0, L.stream>>>(mon, slots[0], slots[1], slots[2], slots[3], out);
    ++*L.counter;
}

template <typename T>
void launch_admission(const Launch& L, const Dom<T>* d_dom, const Dom<T>& h_dom, unsigned long long* d_bad) {
    const int bs = 256;
    k_admission<T><<<(unsigned)((h_dom.ncell + bs - 1) / bs), bs, 0, L.stream>>>(d_dom, d_bad);
    ++*L.counter;
}

void launch_mask_box(const Launch& L, const uint8_t* mask, int nx, int ny, int nz, int* d_box) {
    const int bs = 256;
    const long long n = (long long)nx * ny * nz;
    k_mask_box<<<(unsigned)((n + bs - 1) / bs), bs, 0, L.stream>>>(mask, nx, ny, nz, d_box);
    ++*L.counter;
}

template <typename T>
void launch_nonfinite(const Launch& L, const T* p, long long n, unsigned long long* d_bad) {
    if (n <= 0) return;
    const int bs = 256;
    long long blocks = (n + bs - 1) / bs;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_nonfinite<T><<<(unsigned)blocks, bs, 0, L.stream>>>(p, n, d_bad);
    ++*L.counter;
}

constexpr int kCodecSlabs = 65535;   // slabs of a launch (grid rows)

// Blocks per slab: about 16384 values each, at most a portable cluster.
inline unsigned codec_cluster(long long max_plane) {
    unsigned n = 1;
    while (n < 8 && max_plane / n > 16384) n *= 2;
    return n;
}

template <typename T>
void launch_bf16_encode(const Launch& L, const CodecSeg* segs, int nseg, int nslab, long long max_plane, void* slot) {
    const unsigned n = codec_cluster(max_plane);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kCodecThreads);
    cfg.stream = L.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    for (int first = 0; first < nslab; first += kCodecSlabs) {
        cfg.gridDim = dim3(n, (unsigned)std::min(kCodecSlabs, nslab - first));
        cudaLaunchKernelEx(&cfg, k_bf16_encode<T>, segs, nseg, first, (char*)slot);
        ++*L.counter;
    }
}

template <typename T>
void launch_bf16_decode(const Launch& L, const CodecSeg* segs, int nseg, int nslab, long long max_plane,
                        const void* slot) {
    for (int first = 0; first < nslab; first += kCodecSlabs) {
        const dim3 g(codec_cluster(max_plane), (unsigned)std::min(kCodecSlabs, nslab - first));
        k_bf16_decode<T><<<g, kCodecThreads, 0, L.stream>>>(segs, nseg, first, (const char*)slot);
        ++*L.counter;
    }
}

// Clears an array of 4-byte words, also one in pinned host memory (a host-streamed context's state): the host's own
// memset of a 256^3 state took about 20 ms, this store over the link 2.
__global__ void __launch_bounds__(256) k_zero(unsigned* __restrict__ p, long long n) {
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, dt = (long long)gridDim.x * blockDim.x;
    const long long nv = n >> 2;
    uint4* v = reinterpret_cast<uint4*>(p);
    for (long long t = t0; t < nv; t += dt) v[t] = make_uint4(0u, 0u, 0u, 0u);
    if (t0 < (n & 3)) p[(nv << 2) + t0] = 0u;
}

void launch_zero(const Launch& L, void* p, long long bytes) {
    if (bytes <= 0) return;
    const long long blocks = (bytes / 16 + 255) / 256;
    k_zero<<<(unsigned)std::max(1ll, std::min(blocks, 152ll * 8)), 256, 0, L.stream>>>((unsigned*)p, bytes / 4);
    ++*L.counter;
}

// ---- native snapshots ----------------------------------------------------------------------
// One launch moves every state part between the live arrays and a snapshot slot: block row y
// copies segment y, grid-stride along x.  Slot offsets are 256-byte aligned; a part array starts
// on a 256-byte boundary (fields, CPML memories) or at least on its element size (pole-state parts
// inside one allocation), and its size is a whole number of elements of >= 4 bytes.  16-byte
// vectors where both ends are 16-byte aligned (the last bytes % 16 bytes by lanes of block x = 0),
// 4-byte words otherwise.
__global__ void k_snapshot_copy(const SnapSeg* __restrict__ segs, char* __restrict__ slot, int to_slot) {
    const SnapSeg sg = segs[blockIdx.y];
    const char* src = to_slot ? sg.state : slot + sg.off;
    char* dst = to_slot ? slot + sg.off : sg.state;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, dt = (long long)gridDim.x * blockDim.x;
    if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
        const long long nv = sg.bytes >> 4;
        const int4* s4 = reinterpret_cast<const int4*>(src);
        int4* d4 = reinterpret_cast<int4*>(dst);
        for (long long v = t0; v < nv; v += dt) d4[v] = s4[v];
        const int tail = (int)(sg.bytes & 15);
        if (blockIdx.x == 0 && (int)threadIdx.x < tail) dst[(nv << 4) + threadIdx.x] = src[(nv << 4) + threadIdx.x];
    } else {
        const long long nw = sg.bytes >> 2;
        const unsigned* s1 = reinterpret_cast<const unsigned*>(src);
        unsigned* d1 = reinterpret_cast<unsigned*>(dst);
        for (long long v = t0; v < nw; v += dt) d1[v] = s1[v];
    }
}

void launch_snapshot_copy(const Launch& L, const SnapSeg* segs, int nseg, long long max_bytes, void* slot,
                          int to_slot) {
    if (nseg <= 0) return;
    long long bx = ((max_bytes >> 4) + 256 * 8 - 1) / (256 * 8);   // <= 8 vectors per thread
    bx = bx < 1 ? 1 : (bx > 1024 ? 1024 : bx);
    k_snapshot_copy<<<dim3((unsigned)bx, (unsigned)nseg), 256, 0, L.stream>>>(segs, (char*)slot, to_slot);
    ++*L.counter;
}

#define GBFDTD_INST(T)                                                                                     \
    template void launch_admission<T>(const Launch&, const Dom<T>*, const Dom<T>&, unsigned long long*);   \
    template void launch_nonfinite<T>(const Launch&, const T*, long long, unsigned long long*);             \
    template void launch_bf16_encode<T>(const Launch&, const CodecSeg*, int, int, long long, void*);        \
    template void launch_bf16_decode<T>(const Launch&, const CodecSeg*, int, int, long long, const void*);
GBFDTD_INST(float)
GBFDTD_INST(double)
#undef GBFDTD_INST

}  // namespace gbfdtd
