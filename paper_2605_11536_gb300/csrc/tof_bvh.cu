// tof_bvh.cu -- GPU LBVH for the ToF ReSTIR hot path (sm_103a).
//
// The paper traces rays with DXR hardware BVHs (Sec. 6, Falcor on an RTX 3090); GB300 has no
// RT cores, so visibility runs on a software LBVH built here:
//   xform_kernel    rigid 3x4 object transform of every triangle corner, per frame
//   bounds / morton 30-bit Morton codes of triangle centroids in the centroid bounds (cubic cells)
//   radix sort      4 stable 8-bit LSD passes (tile histograms, offsets, ranked scatter), one cooperative
//                   launch up to 307k triangles
//   karras_kernel   binary radix tree over the sorted codes (Karras, HPG 2012), ties broken by index; lists
//                   the ranges of at most 512 leaves below which it is rebuilt
//   range_box / treelet / treelet_top_kernel   those ranges, and the levels above them, top-down by the surface
//                   area heuristic; leaf records in leaf order
//   refit_kernel    (refits, one triangle) leaf records and bottom-up child boxes of the hierarchy as it is (one
//                   atomic per node; the second arriving thread continues, no thread waits)
//   etree_*_kernel  the ellipsoidal connection's hierarchy over triangle index ranges (boxes and
//                   areas, bottom-up: 8 levels per block in shared memory, then one block)
#include <cstdio>

#include <cooperative_groups.h>

#include "tof_internal.h"

namespace tof {

__device__ __forceinline__ float3 fx3(const float* M, float3 p, int r) {
    (void)r;
    return make_float3(M[0] * p.x + M[1] * p.y + M[2] * p.z + M[3], M[4] * p.x + M[5] * p.y + M[6] * p.z + M[7],
                       M[8] * p.x + M[9] * p.y + M[10] * p.z + M[11]);
}

// per triangle: world corners -> (v0, mat), (e1), (e2); centroid
// (and the empty centroid bounds, encoded minima at 0xFFFFFFFF and maxima at 0, and the number of treelets)
__global__ void xform_kernel(int nt, const float* __restrict__ vloc, const uint32_t* __restrict__ tris,
                             const uint32_t* __restrict__ triobj, const uint32_t* __restrict__ objmat,
                             const float* __restrict__ xf, float4* __restrict__ tri_out, float4* __restrict__ cent,
                             uint32_t* __restrict__ bb) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 7) bb[t] = t < 3 ? 0xFFFFFFFFu : 0u;
    if (t >= nt) return;
    uint32_t o = triobj[t];
    const float* M = xf + 12 * (size_t)o;
    float3 v[3];
    for (int c = 0; c < 3; ++c) {
        uint32_t vi = tris[3 * (size_t)t + c];
        float3 p = make_float3(vloc[3 * (size_t)vi], vloc[3 * (size_t)vi + 1], vloc[3 * (size_t)vi + 2]);
        v[c] = fx3(M, p, 0);
    }
    float3 e1 = make_float3(v[1].x - v[0].x, v[1].y - v[0].y, v[1].z - v[0].z);
    float3 e2 = make_float3(v[2].x - v[0].x, v[2].y - v[0].y, v[2].z - v[0].z);
    tri_out[3 * (size_t)t] = make_float4(v[0].x, v[0].y, v[0].z, __int_as_float((int)objmat[o]));
    tri_out[3 * (size_t)t + 1] = make_float4(e1.x, e1.y, e1.z, 0.f);
    tri_out[3 * (size_t)t + 2] = make_float4(e2.x, e2.y, e2.z, 0.f);
    if (cent) cent[t] = make_float4((v[0].x + v[1].x + v[2].x) / 3.0f, (v[0].y + v[1].y + v[2].y) / 3.0f,
                                    (v[0].z + v[1].z + v[2].z) / 3.0f, 0.f);
}

// order-preserving float <-> uint for atomic min / max
__device__ __forceinline__ uint32_t fenc(float f) {
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fdec(uint32_t u) { return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u); }

__global__ void bounds_kernel(int n, const float4* __restrict__ cent, uint32_t* __restrict__ bb) {
    __shared__ uint32_t s[6];
    if (threadIdx.x < 3) s[threadIdx.x] = 0xFFFFFFFFu;
    else if (threadIdx.x < 6) s[threadIdx.x] = 0u;
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float4 c = cent[i];
        atomicMin(&s[0], fenc(c.x)); atomicMin(&s[1], fenc(c.y)); atomicMin(&s[2], fenc(c.z));
        atomicMax(&s[3], fenc(c.x)); atomicMax(&s[4], fenc(c.y)); atomicMax(&s[5], fenc(c.z));
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(&bb[threadIdx.x], s[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&bb[threadIdx.x], s[threadIdx.x]);
}

__device__ __forceinline__ uint32_t expand10(uint32_t v) {
    v = (v * 0x00010001u) & 0xFF0000FFu;
    v = (v * 0x00000101u) & 0x0F00F00Fu;
    v = (v * 0x00000011u) & 0xC30C30C3u;
    v = (v * 0x00000005u) & 0x49249249u;
    return v;
}

__global__ void morton_kernel(int n, const float4* __restrict__ cent, const uint32_t* __restrict__ bb,
                              uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float lo[3] = {fdec(bb[0]), fdec(bb[1]), fdec(bb[2])}, hi[3] = {fdec(bb[3]), fdec(bb[4]), fdec(bb[5])};
    float4 c = cent[i];
    float cc[3] = {c.x, c.y, c.z};
    uint32_t q[3];
    // one scale for all axes (the largest extent): in a flat scene the top-level splits then cut
    // the long axes, instead of slicing the thin one into wide, flat boxes that every grazing ray
    // crosses (about 11 % lower SAH cost on a 20 m x 12.5 m x 2 m terrain scene)
    const float ext = fmaxf(fmaxf(fmaxf(hi[0] - lo[0], hi[1] - lo[1]), hi[2] - lo[2]), 1e-20f);
    for (int k = 0; k < 3; ++k) {
        float t = (cc[k] - lo[k]) / ext * 1024.0f;
        q[k] = (uint32_t)fminf(fmaxf(t, 0.f), 1023.f);
    }
    keys[i] = (expand10(q[0]) << 2) | (expand10(q[1]) << 1) | expand10(q[2]);
    vals[i] = (uint32_t)i;
}

// ---- radix sort: 2048-key tiles --------------------------------------------------------------
constexpr int kTile = 2048;

__global__ void __launch_bounds__(256) radix_hist_kernel(const uint32_t* __restrict__ keys, int n, int shift,
                                                         uint32_t* __restrict__ hist, int ntiles) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0u;
    __syncthreads();
    int base = blockIdx.x * kTile;
    for (int i = threadIdx.x; i < kTile; i += 256) {
        int g = base + i;
        if (g < n) atomicAdd(&h[(keys[g] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// exclusive scan of a block's 256 values; all = their sum
__device__ __forceinline__ uint32_t scan256(uint32_t x, uint32_t* wsum, uint32_t& all) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
    }
    __syncthreads();   // wsum's last values are read
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t low = 0u;
    all = 0u;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        low += w < warp ? wsum[w] : 0u;
        all += wsum[w];
    }
    return low + incl - x;
}
// one digit's counts over the tiles (row) become each tile's offset within the digit; returns their sum
__device__ __forceinline__ uint32_t scan_digit(uint32_t* row, int ntiles, uint32_t* wsum) {
    uint32_t run = 0u;
    for (int t0 = 0; t0 < ntiles; t0 += 256) {
        const int t = t0 + (int)threadIdx.x;
        uint32_t all;
        const uint32_t before = scan256(t < ntiles ? __ldcg(&row[t]) : 0u, wsum, all);
        if (t < ntiles) row[t] = run + before;
        run += all;
    }
    return run;
}
// a block per digit (one block for all 256 * ntiles counts: 1.74 ms of a 4M-triangle sort's four passes)
__global__ void __launch_bounds__(256) radix_scan_kernel(uint32_t* __restrict__ hist, uint32_t* __restrict__ totals, int ntiles) {
    __shared__ uint32_t wsum[8];
    const uint32_t sum = scan_digit(hist + (size_t)blockIdx.x * ntiles, ntiles, wsum);
    if (threadIdx.x == 0) totals[blockIdx.x] = sum;
}

__global__ void __launch_bounds__(256) radix_scatter_kernel(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                            uint32_t* __restrict__ kout, uint32_t* __restrict__ vout, int n,
                                                            int shift, const uint32_t* __restrict__ offs,
                                                            const uint32_t* __restrict__ totals, int ntiles) {
    __shared__ uint32_t base[256];
    __shared__ uint32_t wsum[8];
    __shared__ uint32_t wc[8][256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t all;
    base[tid] = scan256(totals[tid], wsum, all) + offs[(size_t)tid * ntiles + blockIdx.x];
    const uint32_t lt = (1u << lane) - 1u;
    for (int r = 0; r < kTile / 256; ++r) {
        for (int k = 0; k < 8; ++k) wc[k][tid] = 0u;
        __syncthreads();
        int i = blockIdx.x * kTile + r * 256 + tid;
        bool valid = i < n;
        uint32_t key = valid ? kin[i] : 0u;
        uint32_t dg = (key >> shift) & 255u;
        uint32_t peers = __match_any_sync(0xFFFFFFFFu, valid ? dg : 256u + (uint32_t)lane);
        uint32_t rank = __popc(peers & lt);
        if (valid && rank == 0) wc[warp][dg] = __popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t off = base[dg] + rank;
            for (int w = 0; w < warp; ++w) off += wc[w][dg];
            kout[off] = key;
            vout[off] = vin[i];
        }
        __syncthreads();
        uint32_t tot = 0;
        for (int w = 0; w < 8; ++w) tot += wc[w][tid];
        base[tid] += tot;
        __syncthreads();
    }
}

// The same four passes in one cooperative launch of one block per tile of 512 keys (all resident): per
// pass the tile histograms, a grid-wide sync, each tile's digit offsets, the same stable scatter, and a
// grid-wide sync.  Sorted keys and values are those of the separate launches (after four passes back in k0 / v0).
// Bound by the latency of its barriers and dependent steps: a tile of 512 keys has two ranking rounds a pass
// where one of 2048 has eight, and its keys stay in registers from the histogram to the scatter.  Offsets:
// every block adds up all tiles' histograms itself, or (kScan) the digits' rows are scanned by a block
// each, a third grid-wide sync for a time that does not grow with the tiles (kAddTiles).
constexpr int kCoopTile = 512;
template <bool kScan>
__global__ void __launch_bounds__(256) radix_sort_coop_kernel(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, int n,
                                                              uint32_t* __restrict__ hist, int ntiles) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    constexpr int kRounds = kCoopTile / 256;
    __shared__ uint32_t h[256];
    __shared__ uint32_t base[256];
    __shared__ uint32_t wc[8][256];
    __shared__ uint32_t wsum[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t *ki = k0, *vi = v0, *ko = k1, *vo = v1;
    uint32_t* const totals = hist + (size_t)256 * ntiles;   // kScan
    const int t0 = blockIdx.x * kCoopTile;
    for (int shift = 0; shift < 32; shift += 8) {
        h[tid] = 0u;
        __syncthreads();
        uint32_t key[kRounds];
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            const int g = t0 + r * 256 + tid;
            key[r] = g < n ? __ldcg(&ki[g]) : 0u;
            if (g < n) atomicAdd(&h[(key[r] >> shift) & 255u], 1u);
        }
        __syncthreads();
        hist[kScan ? (size_t)tid * ntiles + blockIdx.x : (size_t)blockIdx.x * 256 + tid] = h[tid];
        __threadfence();
        grid.sync();
        uint32_t tot = 0u, before = 0u, all;
        if constexpr (kScan) {
            for (int d = blockIdx.x; d < 256; d += gridDim.x) {
                const uint32_t sum = scan_digit(hist + (size_t)d * ntiles, ntiles, wsum);
                if (tid == 0) totals[d] = sum;
            }
            __threadfence();
            grid.sync();
            tot = __ldcg(&totals[tid]);
            before = __ldcg(&hist[(size_t)tid * ntiles + blockIdx.x]);
        } else {
#pragma unroll 8
            for (int t = 0; t < ntiles; ++t) {
                const uint32_t c = __ldcg(&hist[t * 256 + tid]);
                tot += c;
                if (t < (int)blockIdx.x) before += c;
            }
        }
        base[tid] = scan256(tot, wsum, all) + before;
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            for (int k = 0; k < 8; ++k) wc[k][tid] = 0u;
            __syncthreads();
            const int i = t0 + r * 256 + tid;
            const bool valid = i < n;
            const uint32_t val = valid ? __ldcg(&vi[i]) : 0u;
            const uint32_t dg = (key[r] >> shift) & 255u;
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, valid ? dg : 256u + (uint32_t)lane);
            const uint32_t rank = __popc(peers & lt);
            if (valid && rank == 0) wc[warp][dg] = __popc(peers);
            __syncthreads();
            if (valid) {
                uint32_t off = base[dg] + rank;
                for (int w = 0; w < warp; ++w) off += wc[w][dg];
                ko[off] = key[r];
                vo[off] = val;
            }
            if (r + 1 < kRounds) {
                __syncthreads();
                uint32_t add = 0;
                for (int w = 0; w < 8; ++w) add += wc[w][tid];
                base[tid] += add;
                __syncthreads();
            }
        }
        __threadfence();
        grid.sync();
        uint32_t* t = ki; ki = ko; ko = t;
        t = vi; vi = vo; vo = t;
    }
}

// ---- Karras 2012 hierarchy --------------------------------------------------------------------
__device__ __forceinline__ int delta(const uint32_t* __restrict__ k, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    uint32_t a = k[i], b = k[j];
    if (a == b) return 32 + __clz((uint32_t)i ^ (uint32_t)j);
    return __clz(a ^ b);
}

// Ranges of at most kTreelet leaves whose parent's is larger are listed as treelets (cuts[r] = (first leaf,
// leaves | kRootLast where the Karras node of the range is numbered by its last leaf), *ncut of them).
constexpr int kTreelet = 512;
constexpr int kWhole = 1024;   // a scene of so many triangles is one range (whole_kernel)
constexpr uint32_t kRootLast = 0x80000000u;
__device__ __forceinline__ void list_cut(int first, int last, int code, uint32_t* __restrict__ cut_a, uint32_t* __restrict__ cut_m,
                                         uint32_t* ncut) {
    const uint32_t r = atomicAdd(ncut, 1u);
    cut_a[r] = (uint32_t)first;
    cut_m[r] = (uint32_t)(last - first + 1) | (code == last && last > first ? kRootLast : 0u);
}
__global__ void karras_kernel(int n, const uint32_t* __restrict__ keys, int* __restrict__ child, int* __restrict__ parent_int,
                              int* __restrict__ parent_leaf, uint32_t* __restrict__ cut_a, uint32_t* __restrict__ cut_m,
                              uint32_t* ncut, uint32_t* __restrict__ counter) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    if (counter) counter[i] = 0u;
    int d = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = delta(keys, n, i, i - d);
    int lmax = 2;
    while (delta(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
    int j = i + l * d;
    int dnode = delta(keys, n, i, j);
    int s = 0;
    int div = 2;
    int t = (l + div - 1) / div;
    while (true) {
        if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
        if (t == 1) break;
        div <<= 1;
        t = (l + div - 1) / div;
    }
    int g = i + s * d + (d < 0 ? -1 : 0);
    int left = min(i, j) == g ? ~g : g;
    int right = max(i, j) == g + 1 ? ~(g + 1) : g + 1;
    child[2 * i] = left;
    child[2 * i + 1] = right;
    if (left < 0) parent_leaf[~left] = i; else parent_int[left] = i;
    if (right < 0) parent_leaf[~right] = i; else parent_int[right] = i;
    if (i == 0) parent_int[0] = -1;
    const int first = min(i, j), last = max(i, j);
    if (last - first + 1 > kTreelet) {
        if (g - first + 1 <= kTreelet) list_cut(first, g, left, cut_a, cut_m, ncut);
        if (last - g <= kTreelet) list_cut(g + 1, last, right, cut_a, cut_m, ncut);
    }
}

struct Box { float lo[3], hi[3]; };

__device__ __forceinline__ Box tri_box(const float4* __restrict__ tri, int t) {
    float4 a = tri[3 * (size_t)t], e1 = tri[3 * (size_t)t + 1], e2 = tri[3 * (size_t)t + 2];
    float v[3][3] = {{a.x, a.y, a.z}, {a.x + e1.x, a.y + e1.y, a.z + e1.z}, {a.x + e2.x, a.y + e2.y, a.z + e2.z}};
    Box b;
    for (int k = 0; k < 3; ++k) {
        float lo = fminf(v[0][k], fminf(v[1][k], v[2][k])), hi = fmaxf(v[0][k], fmaxf(v[1][k], v[2][k]));
        float pad = 1e-6f * fmaxf(fabsf(lo), fabsf(hi)) + 1e-6f;   // conservative against rounding
        b.lo[k] = lo - pad; b.hi[k] = hi + pad;
    }
    return b;
}
__device__ __forceinline__ Box node_box(const float4* N) {
    float4 n0 = __ldcg(N), n1 = __ldcg(N + 1), n2 = __ldcg(N + 2);
    Box b;
    b.lo[0] = fminf(n0.x, n1.x); b.hi[0] = fmaxf(n0.y, n1.y);
    b.lo[1] = fminf(n0.z, n1.z); b.hi[1] = fmaxf(n0.w, n1.w);
    b.lo[2] = fminf(n2.x, n2.z); b.hi[2] = fmaxf(n2.y, n2.w);
    return b;
}

// arrival counter of a node: acquire-release at device scope, so that the second arrival sees the
// node the first arrival wrote below it (release of its writes, acquire of the sibling's)
__device__ __forceinline__ uint32_t arrive_acq_rel(uint32_t* p) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
    return old;
}

__global__ void refit_kernel(int n, const uint32_t* __restrict__ prim, const float4* __restrict__ tri, float4* __restrict__ leaf,
                             float4* nodes, const int* __restrict__ child, const int* __restrict__ parent_int,
                             const int* __restrict__ parent_leaf, uint32_t* __restrict__ counter) {
    int L = blockIdx.x * blockDim.x + threadIdx.x;
    if (L >= n) return;
    int t = (int)prim[L];
    float4 a = tri[3 * (size_t)t];
    leaf[3 * (size_t)L] = make_float4(a.x, a.y, a.z, __int_as_float(t));
    leaf[3 * (size_t)L + 1] = tri[3 * (size_t)t + 1];
    leaf[3 * (size_t)L + 2] = tri[3 * (size_t)t + 2];
    if (n == 1) return;
    int p = parent_leaf[L];
    int guard = n;   // depth of a valid hierarchy is below n
    while (p >= 0 && --guard >= 0) {
        if (arrive_acq_rel(&counter[p]) == 0u) return;   // first arrival: the sibling finishes p
        int c[2] = {child[2 * p], child[2 * p + 1]};
        Box b[2];
        for (int k = 0; k < 2; ++k) b[k] = c[k] < 0 ? tri_box(tri, (int)prim[~c[k]]) : node_box(nodes + 4 * (size_t)c[k]);
        float4* N = nodes + 4 * (size_t)p;
        N[0] = make_float4(b[0].lo[0], b[0].hi[0], b[0].lo[1], b[0].hi[1]);
        N[1] = make_float4(b[1].lo[0], b[1].hi[0], b[1].lo[1], b[1].hi[1]);
        N[2] = make_float4(b[0].lo[2], b[0].hi[2], b[1].lo[2], b[1].hi[2]);
        N[3] = make_float4(__int_as_float(c[0]), __int_as_float(c[1]), 0.f, 0.f);
        p = parent_int[p];
    }
}

// ---- surface-area treelets ---------------------------------------------------------------------
// A Morton-code hierarchy splits space in halves whatever lies in them: rays visit 1.25 to 2 times the
// nodes that they do in one split by the surface area heuristic (host model, visits per ray: terrain with
// spheres 36 against 29 for bounce rays and 40 against 31 for visibility, full top-down SAH 27 and 29;
// confocal scan 18 against 11.5; box 13.6 against 7.2).  So the Morton order is cut into ranges of at most
// 512 leaves, each is built anew top-down by one block -- every split of the sorted orders tried, all nodes
// of a level at once, the triangles' boxes in shared memory -- and one block builds the levels above over
// the ranges' boxes in the same way, beside them (up to 1024 of them; more keep the Morton hierarchy there).
// Frames with the build: 512 x 512 2.73 -> 2.63 ms, 1024 x 1024 11.1 -> 10.4; static scenes: path tracing 608 ->
// 446 us, 128 x 128 allocation-free 428 -> 361 us.  A build alone, us, bottom-up boxes of the Morton hierarchy / first
// form of this / now: 312 triangles 87 / 130 / 63, 968 101 / 116 / 80, 5000 130 / 119 / 104, 66k 163 / 169 / 150, 198k 214 /
// 304 / 205, 270k 266 / 392 / 271, 646k 819 / 807 / 499, 4M 2629 / 4850 / 2090.
// It writes boxes, children and leaf order itself, so a full build needs no bottom-up pass over all levels.
// Node numbers: a range [a, a + m) owns the m - 1 numbers of its Karras nodes; its root keeps the Karras
// root's, so that a Karras parent's link to it stays right.
template <int N>
struct Sweep {
    float box[6][N];                  // lo, hi of item i
    uint32_t keys[3][N];              // the sort's exchange
    unsigned long long best[N];       // per segment start: (cost and distance from the middle, axis, position)
    uint16_t ord[3][N];               // items sorted along each axis within their segment
    uint16_t seg0[N], seg1[N];        // segment [seg0, seg1) of a position
    uint8_t side[N];                  // of an item: right of its segment's split
    int link[N];                      // per segment start: 2 * parent + side of the node to come, or -1
    float wup[3][N / 32][6], wdown[3][N / 32][6];
    uint32_t bal[3][N / 32];          // per warp and axis: the positions whose item goes left
    int root_split, open[2];          // open: leaves of the longest segment to split, by the level's parity
};
__device__ __forceinline__ float half_area(const float b[6]) {
    const float x = b[3] - b[0], y = b[4] - b[1], z = b[5] - b[2];
    return x * y + y * z + z * x;
}
__device__ __forceinline__ void grow(float b[6], const float o[6]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) { b[k] = fminf(b[k], o[k]); b[3 + k] = fmaxf(b[3 + k], o[3 + k]); }
}
// barrier of the block's first nt threads (a multiple of 32): a range shorter than the block's threads
// leaves the other warps out
__device__ __forceinline__ void group_sync(int nt) { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); }
// the running box of a lane's segment within its warp, over the `before` lanes below it that are in the segment
// (kUp) or the `before` lanes above it
template <bool kUp>
__device__ __forceinline__ void run_boxes(int reach, int before, float b[6]) {
#pragma unroll 1
    for (int o = 1; o < 32 && o < reach; o <<= 1) {
        float n[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) n[k] = kUp ? __shfl_up_sync(0xFFFFFFFFu, b[k], o) : __shfl_down_sync(0xFFFFFFFFu, b[k], o);
        if (before >= o) grow(b, n);
    }
}

// Builds the hierarchy of items 0 .. m - 1 (m >= 2, boxes in S.box) with N threads.  number(split,
// root_split) is the node that splits after position `split`; leaf(position, item) the child code of one item;
// up(code, node) records a child's parent.  Levels from `sweeps` on split in the middle, which bounds the
// depth (coincident items): 16 and 10 levels in a range of 512, 16 and 11 above 1024 ranges, 53 of the 64 that a
// traversal's stack holds.  Below the Morton hierarchy's own top, which can be 30 levels and the logarithm of its
// ranges deep, 8 and 10 levels.  kAll: every split of the three orders is tried, else those of the order along
// the segment's longest axis (a third of the work, visits per ray up 2 %; a scene of at most 512 triangles
// tries all, 12 % fewer visits in the 332-triangle box).
// Bound by issue (62 % active with three blocks an SM; some 10k instructions a warp over about 14 levels, a third of
// them the running boxes) and its chain of barriers, so: the three orders are sorted together, keys in
// registers, barriers only for exchanges between warps; a level has five barriers (eleven at first); the best
// split of a segment is found by shuffles with one shared atomic for each warp and segment; 40 registers.
// treelet_kernel 66k triangles 71 -> 57 us, 198k 130 -> 93, 4M 2.08 -> 1.52 ms.
constexpr int kMaxSweep = 16, kMortonSweep = 8;
template <int N, bool kAll, class Number, class Leaf, class Up>
__device__ __forceinline__ void sweep_build(Sweep<N>& S, int m, int sweeps, float4* __restrict__ nodes, int* __restrict__ child, Number number, Leaf leaf,
                                            Up up) {
    const int p = threadIdx.x, lane = p & 31, warp = p >> 5;
    int pow2 = 32;
    while (pow2 < m) pow2 <<= 1;
    if (p >= pow2) return;
    {   // centre (in 2^22 steps of the items' extent), then item: an order of all items along each axis (bitonic
        // sort; padding sorts last)
        uint32_t key[3];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const float c = p < m ? S.box[ax][p] + S.box[3 + ax][p] : 0.f;
            const uint32_t lo = __reduce_min_sync(0xFFFFFFFFu, p < m ? fenc(c) : 0xFFFFFFFFu);
            const uint32_t hi = __reduce_max_sync(0xFFFFFFFFu, p < m ? fenc(c) : 0u);
            if (lane == 0) { S.keys[ax][warp] = lo; S.keys[ax][N / 2 + warp] = hi; }
        }
        group_sync(pow2);
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const uint32_t lo = __reduce_min_sync(0xFFFFFFFFu, lane < pow2 / 32 ? S.keys[ax][lane] : 0xFFFFFFFFu);
            const uint32_t hi = __reduce_max_sync(0xFFFFFFFFu, lane < pow2 / 32 ? S.keys[ax][N / 2 + lane] : 0u);
            const float c = p < m ? S.box[ax][p] + S.box[3 + ax][p] : 0.f, l = fdec(lo), w = fdec(hi) - l;
            const uint32_t q = (uint32_t)fminf(fmaxf((c - l) / fmaxf(w, 1e-30f) * 4194304.f, 0.f), 4194302.f);
            key[ax] = p < m ? (q << 10) | (uint32_t)p : 0xFFFFFFFFu;
        }
        group_sync(pow2);
#pragma unroll 1
        for (int k = 2; k <= pow2; k <<= 1)
#pragma unroll 1
            for (int j = k >> 1; j > 0; j >>= 1) {
                const bool low = ((p & k) == 0) == ((p & j) == 0);   // this place keeps the lower key
                uint32_t o[3];
                if (j >= 32) {
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) S.keys[ax][p] = key[ax];
                    group_sync(pow2);
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) o[ax] = S.keys[ax][p ^ j];
                    group_sync(pow2);
                } else {
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) o[ax] = __shfl_xor_sync(0xFFFFFFFFu, key[ax], j);
                }
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) key[ax] = low ? min(key[ax], o[ax]) : max(key[ax], o[ax]);
            }
        if (p < m)
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) S.ord[ax][p] = (uint16_t)(key[ax] & 1023u);
    }
    const int nt = (m + 31) & ~31;
    if (p >= nt) return;
    if (p < m) { S.seg0[p] = 0; S.seg1[p] = (uint16_t)m; }
    if (p == 0) { S.link[0] = -1; S.root_split = -1; S.open[0] = m; S.best[0] = ~0ull; }
    group_sync(nt);
#pragma unroll 1
    for (int level = 0;; ++level) {
        if (S.open[level & 1] <= 1) break;   // leaves of the longest segment
        if (p == 0) S.open[(level + 1) & 1] = 0;
        const int s = p < m ? S.seg0[p] : 0, e = p < m ? S.seg1[p] : 0;
        const bool in = e - s > 1;   // a segment to split
        // lanes of the segment below and above this one in the warp
        const int below = in ? min(lane, p - s) : 0, above = in ? min(31 - lane, e - 1 - p) : 0;
        const int reach = __reduce_max_sync(0xFFFFFFFFu, in ? e - s : 0);   // the warp's longest segment
        if (reach == 0) {   // none in this warp: it only keeps the barriers' count
#pragma unroll 1
            for (int t = 0; t < (kAll ? 7 : 5); ++t) group_sync(nt);
            continue;
        }
        float L[6], R[6], cost = 3.4e38f;
        int axis = 0, item = 0;
        bool any = false;
        if (!kAll && e - s > 2) {   // (of two items every order gives the same split)
            // by the centres: by the sides of the segment's box the build is 8 us shorter (198k triangles), but a
            // 301 x 203 frame 20 us longer
            float ext = -1.0f;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                const int i0 = S.ord[ax][s], i1 = S.ord[ax][e - 1];
                const float x = (S.box[ax][i1] + S.box[3 + ax][i1]) - (S.box[ax][i0] + S.box[3 + ax][i0]);
                if (x > ext) { ext = x; axis = ax; }
            }
        }
#pragma unroll 1
        for (int t = 0; t < (kAll ? 3 : 1); ++t) {
            const int ax = kAll ? t : axis;
            float f[6], b[6];
            item = in ? S.ord[ax][p] : 0;
#pragma unroll
            for (int k = 0; k < 6; ++k) b[k] = f[k] = S.box[k][item];
            run_boxes<true>(reach, below, f);
            run_boxes<false>(reach, above, b);
            // across warps: a segment's part in each warp it reaches over
            if (lane == 31)
#pragma unroll
                for (int k = 0; k < 6; ++k) S.wup[t][warp][k] = f[k];
            if (lane == 0)
#pragma unroll
                for (int k = 0; k < 6; ++k) S.wdown[t][warp][k] = b[k];
            group_sync(nt);
            // b becomes the box of the positions behind p
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                b[k] = __shfl_down_sync(0xFFFFFFFFu, b[k], 1);
                if (lane == 31) b[k] = k < 3 ? 3.4e38f : -3.4e38f;
            }
            if (in) {
                for (int v = warp - 1; v >= 0 && 32 * v + 31 >= s; --v) grow(f, S.wup[t][v]);
                for (int v = warp + 1; 32 * v < e; ++v) grow(b, S.wdown[t][v]);
                if (p + 1 < e) {
                    const float c = level >= sweeps ? 0.f : half_area(f) * (float)(p + 1 - s) + half_area(b) * (float)(e - 1 - p);
                    if (!any || c < cost) {
                        any = true;
                        cost = c; axis = ax;
#pragma unroll
                        for (int k = 0; k < 6; ++k) { L[k] = f[k]; R[k] = b[k]; }
                    }
                }
            }
        }
        // the split's cost to 18 bits, of equals the one nearest to the middle
        uint32_t key = 0xFFFFFFFFu;
        if (any) key = (__float_as_uint(cost) & ~63u) | (uint32_t)min(63, abs(2 * (p + 1 - s) - (e - s)) >> (31 - __clz(e - s) > 6 ? 25 - __clz(e - s) : 0));
        uint32_t low = key;
#pragma unroll 1
        for (int o = 1; o < 32 && o < reach; o <<= 1) {
            const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, low, o);
            if (below >= o) low = min(low, n);
        }
        low = __shfl_sync(0xFFFFFFFFu, low, lane + above);   // of the segment's part in this warp
        const uint32_t same = __ballot_sync(0xFFFFFFFFu, any && key == low) & (0xFFFFFFFFu >> (31 - below - above) << (lane - below));
        if (any && same && __ffs(same) - 1 == lane)
            atomicMin(&S.best[s], ((unsigned long long)key << 32) | (uint32_t)(axis << 10) | (uint32_t)p);
        group_sync(nt);
        const unsigned long long best = in ? S.best[s] : 0ull;
        const int cut = (int)(best & 1023u);   // the segment splits after this position of its axis' order
        if (in) S.side[kAll ? S.ord[(best >> 10) & 3u][p] : item] = p > cut;
        if (in && p == cut) {
            if (level == 0) S.root_split = p;
            const int id = number(p, level == 0 ? p : S.root_split);
            nodes[4 * (size_t)id] = make_float4(L[0], L[3], L[1], L[4]);
            nodes[4 * (size_t)id + 1] = make_float4(R[0], R[3], R[1], R[4]);
            nodes[4 * (size_t)id + 2] = make_float4(L[2], L[5], R[2], R[5]);
            const int link = S.link[s];
            if (link >= 0) {
                child[link] = id;
                reinterpret_cast<int*>(nodes + 4 * (size_t)(link >> 1) + 3)[link & 1] = id;
                up(id, link >> 1);
            }
            S.link[s] = 2 * id;        // an open left part keeps the start
            S.link[p + 1] = 2 * id + 1;
        }
        group_sync(nt);
        // stable partition of the three orders
        int part[3];
        uint32_t bal[3];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            part[ax] = in ? S.ord[ax][p] : 0;
            const bool l = in && S.side[part[ax]] == 0;
            bal[ax] = __ballot_sync(0xFFFFFFFFu, l);
            if (lane == 0) S.bal[ax][warp] = bal[ax];
        }
        group_sync(nt);
        int ns = s, ne = e;
        if (in) {
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                int l = __popc(bal[ax] & ((1u << lane) - (1u << (lane - below))));   // of the left side before this position
                if (s < 32 * warp) {
                    l += __popc(S.bal[ax][s >> 5] >> (s & 31));
                    for (int v = (s >> 5) + 1; v < warp; ++v) l += __popc(S.bal[ax][v]);
                }
                const int dst = (bal[ax] >> lane) & 1u ? s + l : cut + 1 + (p - s) - l;
                S.ord[ax][dst] = (uint16_t)part[ax];
                if (ax == 0) {
                    const int ds = dst <= cut ? s : cut + 1, de = dst <= cut ? cut + 1 : e;
                    if (de - ds == 1) {   // one item left: a child of the node just written
                        const int link = S.link[dst];
                        const int code = leaf(dst, part[0]);
                        child[link] = code;
                        reinterpret_cast<int*>(nodes + 4 * (size_t)(link >> 1) + 3)[link & 1] = code;
                        up(code, link >> 1);
                    }
                }
            }
            ns = p <= cut ? s : cut + 1;
            ne = p <= cut ? cut + 1 : e;
            S.seg0[p] = (uint16_t)ns;
            S.seg1[p] = (uint16_t)ne;
            if (p == ns) S.best[p] = ~0ull;
        }
        const int most = __reduce_max_sync(0xFFFFFFFFu, in ? ne - ns : 0);
        if (lane == 0 && most > 1) atomicMax(&S.open[(level + 1) & 1], most);
        group_sync(nt);
    }
}

// the boxes of at most kTopItems ranges, one block of 128 per range (boxes[2 r], boxes[2 r + 1])
constexpr int kTopItems = 1024;
__device__ __forceinline__ bool top_by_area(int R, int n) { return R > 1 && R <= kTopItems && 2 * R <= n; }
__global__ void __launch_bounds__(128) range_box_kernel(int n, const uint32_t* __restrict__ prim, const float4* __restrict__ tri,
                                                        float4* __restrict__ boxes, const uint32_t* __restrict__ cut_a,
                                                        const uint32_t* __restrict__ cut_m, const uint32_t* __restrict__ ncut) {
    __shared__ float part[4][6];
    const int R = (int)*ncut;
    if (!top_by_area(R, n)) return;
    const int p = threadIdx.x;
    for (int r = blockIdx.x; r < R; r += gridDim.x) {
        const int a = (int)cut_a[r], m = (int)(cut_m[r] & ~kRootLast);
        float b[6] = {3.4e38f, 3.4e38f, 3.4e38f, -3.4e38f, -3.4e38f, -3.4e38f};
#pragma unroll
        for (int i = 0; i < kTreelet / 128; ++i)
            if (128 * i + p < m) {
                const Box t = tri_box(tri, (int)prim[a + 128 * i + p]);
#pragma unroll
                for (int k = 0; k < 3; ++k) { b[k] = fminf(b[k], t.lo[k]); b[3 + k] = fmaxf(b[3 + k], t.hi[k]); }
            }
#pragma unroll
        for (int k = 0; k < 6; ++k)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float x = __shfl_xor_sync(0xFFFFFFFFu, b[k], o);
                b[k] = k < 3 ? fminf(b[k], x) : fmaxf(b[k], x);
            }
        if ((p & 31) == 0)
#pragma unroll
            for (int k = 0; k < 6; ++k) part[p >> 5][k] = b[k];
        __syncthreads();
        if (p == 0) {
            for (int v = 1; v < 4; ++v) grow(b, part[v]);
            boxes[2 * r] = make_float4(b[0], b[1], b[2], 0.f);
            boxes[2 * r + 1] = make_float4(b[3], b[4], b[5], 0.f);
        }
        __syncthreads();
    }
}

// one range: items p = 0 .. m - 1 are the triangles t, leaves a .. a + m - 1
template <int N, bool kAll>
__device__ __forceinline__ void build_range(Sweep<N>& S, int a, int m, bool last, int t, int sweeps, uint32_t* __restrict__ prim,
                                            const float4* __restrict__ tri, float4* __restrict__ leaves, float4* __restrict__ nodes,
                                            int* __restrict__ child, int* __restrict__ parent_int, int* __restrict__ parent_leaf) {
    const int p = threadIdx.x;
    if (p < m) {
        const Box b = tri_box(tri, t);
#pragma unroll
        for (int k = 0; k < 3; ++k) { S.box[k][p] = b.lo[k]; S.box[3 + k][p] = b.hi[k]; }
    }
    __syncthreads();
    int pos = p;   // item p's leaf within the range
    if (m > 1) {
        // numbers a .. a + m - 1 without the end that is not the root's
        const int base = last ? a + 1 : a, root = last ? a + m - 1 : a, at_root = root - base;
        sweep_build<N, kAll>(
            S, m, sweeps, nodes, child,
            [=](int split, int rs) { return split == rs ? root : split == at_root ? base + rs : base + split; },
            [=](int q, int) { return ~(a + q); },
            [=](int code, int node) {
                if (code < 0) parent_leaf[~code] = node;
                else parent_int[code] = node;
            });
        if (p < m) S.seg0[S.ord[0][p]] = (uint16_t)p;
        __syncthreads();
        if (p < m) pos = S.seg0[p];
    }
    if (p < m) {
        const size_t l = (size_t)(a + pos);
        prim[l] = (uint32_t)t;
        const float4 v = tri[3 * (size_t)t];
        leaves[3 * l] = make_float4(v.x, v.y, v.z, __int_as_float(t));
        leaves[3 * l + 1] = tri[3 * (size_t)t + 1];
        leaves[3 * l + 2] = tri[3 * (size_t)t + 2];
    }
}

constexpr int kTreeletBlocks = 3;   // resident on an SM
__global__ void __launch_bounds__(kTreelet, kTreeletBlocks) treelet_kernel(int n, uint32_t* __restrict__ prim, const float4* __restrict__ tri,
                                                           float4* __restrict__ leaves, float4* __restrict__ nodes, int* __restrict__ child,
                                                           int* __restrict__ parent_int, int* __restrict__ parent_leaf,
                                                           const uint32_t* __restrict__ cut_a, const uint32_t* __restrict__ cut_m,
                                                           const uint32_t* __restrict__ ncut) {
    extern __shared__ __align__(16) unsigned char sm[];
    Sweep<kTreelet>& S = *reinterpret_cast<Sweep<kTreelet>*>(sm);
    const uint32_t R = *ncut;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // treelet_top_kernel may start beside this one
    const int sweeps = top_by_area((int)R, n) ? kMaxSweep : kMortonSweep;
    for (uint32_t r = blockIdx.x; r < R; r += gridDim.x) {
        const int a = (int)cut_a[r], m = (int)(cut_m[r] & ~kRootLast);
        const int t = (int)threadIdx.x < m ? (int)prim[a + threadIdx.x] : 0;
        build_range<kTreelet, false>(S, a, m, (cut_m[r] & kRootLast) != 0u, t, sweeps, prim, tri, leaves, nodes, child, parent_int, parent_leaf);
        __syncthreads();
    }
}

// A scene of at most N triangles is one range, built from the triangles as they are: no Morton codes, sort or
// Karras pass (684 triangles: 58 us of kernels against 140 with them, 82 with the bottom-up pass).
template <int N, bool kAll>
__global__ void __launch_bounds__(N) whole_kernel(int n, uint32_t* __restrict__ prim, const float4* __restrict__ tri, float4* __restrict__ leaves,
                                                  float4* __restrict__ nodes, int* __restrict__ child, int* __restrict__ parent_int,
                                                  int* __restrict__ parent_leaf) {
    extern __shared__ __align__(16) unsigned char sm[];
    Sweep<N>& S = *reinterpret_cast<Sweep<N>*>(sm);
    const int p = threadIdx.x;
    if (p == 0) parent_int[0] = -1;
    build_range<N, kAll>(S, 0, n, false, p < n ? p : 0, kMaxSweep, prim, tri, leaves, nodes, child, parent_int, parent_leaf);
}

// The levels above the treelets, one block.  It starts beside treelet_kernel (programmatic launch): the ranges'
// boxes come from range_box_kernel, which is complete when treelet_kernel starts, and the nodes, children and
// parents that the two write are not the same ones.  It ends after treelet_kernel has (every path waits), so
// what follows it in the stream finds both.  Both are chains of short barriers on few SMs (66k triangles: 57 and
// 29 us), so side by side they take little more than the longer: 301 x 203 frame 1.311 -> 1.284 ms, four served
// streams 6.39 -> 6.28, the boxes' own launch included.
// Of more than kTopItems ranges the Morton hierarchy's own nodes above stay, their boxes found bottom-up as in
// refit_kernel: by treelet_top_kernel's block in a scene of up to kClimbBlock triangles, by morton_top_kernel
// in a larger one (4M triangles: 753 us in one block).
constexpr int kClimbBlock = 1 << 18;
__device__ __forceinline__ void climb_range(int r, int n, const uint32_t* prim, const float4* __restrict__ tri, float4* nodes, const int* child,
                                            const int* parent_int, const int* parent_leaf, uint32_t* counter,
                                            const uint32_t* __restrict__ cut_a, const uint32_t* __restrict__ cut_m) {
    const int a = (int)cut_a[r], m = (int)(cut_m[r] & ~kRootLast);
    int q = m == 1 ? parent_leaf[a] : parent_int[(cut_m[r] & kRootLast) ? a + m - 1 : a];
    int guard = n;
    while (q >= 0 && --guard >= 0) {
        if (arrive_acq_rel(&counter[q]) == 0u) break;
        const int c[2] = {child[2 * q], child[2 * q + 1]};
        Box b[2];
        for (int k = 0; k < 2; ++k) b[k] = c[k] < 0 ? tri_box(tri, (int)prim[~c[k]]) : node_box(nodes + 4 * (size_t)c[k]);
        float4* N = nodes + 4 * (size_t)q;
        N[0] = make_float4(b[0].lo[0], b[0].hi[0], b[0].lo[1], b[0].hi[1]);
        N[1] = make_float4(b[1].lo[0], b[1].hi[0], b[1].lo[1], b[1].hi[1]);
        N[2] = make_float4(b[0].lo[2], b[0].hi[2], b[1].lo[2], b[1].hi[2]);
        N[3] = make_float4(__int_as_float(c[0]), __int_as_float(c[1]), 0.f, 0.f);
        q = parent_int[q];
    }
}
__device__ __forceinline__ void wait_for_treelets() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__global__ void __launch_bounds__(kTopItems) treelet_top_kernel(int n, const uint32_t* prim, const float4* __restrict__ tri,
                                                                const float4* __restrict__ boxes, float4* nodes, int* child,
                                                                int* parent_int, int* parent_leaf, uint32_t* counter,
                                                                const uint32_t* __restrict__ cut_a, const uint32_t* __restrict__ cut_m,
                                                                const uint32_t* __restrict__ ncut, bool climb) {
    extern __shared__ __align__(16) unsigned char sm[];
    Sweep<kTopItems>& S = *reinterpret_cast<Sweep<kTopItems>*>(sm);
    __shared__ int s_no_slot, s_slot0;   // the item without a free number; the item whose free number is 0
    const int p = threadIdx.x;
    const int R = (int)*ncut;
    if (top_by_area(R, n)) {
        if (p < R) {
            const int a = (int)cut_a[p], m = (int)(cut_m[p] & ~kRootLast);
            const bool last = (cut_m[p] & kRootLast) != 0u;
            const float4 lo = boxes[2 * p], hi = boxes[2 * p + 1];
            S.box[0][p] = lo.x; S.box[1][p] = lo.y; S.box[2][p] = lo.z;
            S.box[3][p] = hi.x; S.box[4][p] = hi.y; S.box[5][p] = hi.z;
            const int slot = last ? a : a + m - 1;   // the number of the range that none of its nodes has
            if (slot == n - 1) s_no_slot = p;
            if (slot == 0) s_slot0 = p;
        }
        __syncthreads();
        const int none = s_no_slot, zero = s_slot0;
        // R - 1 splits onto the R - 1 free numbers, the root's being 0
        auto slot_item = [=](int split) { return split == none ? R - 1 : split; };
        auto slot_of = [=](int item) { return (cut_m[item] & kRootLast) ? (int)cut_a[item] : (int)(cut_a[item] + (cut_m[item] & ~kRootLast)) - 1; };
        const int zero_split = zero == R - 1 ? none : zero;
        sweep_build<kTopItems, false>(
            S, R, kMaxSweep, nodes, child,
            [=](int split, int rs) { return split == rs ? 0 : slot_of(slot_item(split == zero_split ? rs : split)); },
            [=](int, int item) {
                const int a = (int)cut_a[item], m = (int)(cut_m[item] & ~kRootLast);
                return m == 1 ? ~a : (cut_m[item] & kRootLast) ? a + m - 1 : a;
            },
            [=](int code, int node) {
                if (code < 0) parent_leaf[~code] = node;
                else parent_int[code] = node;
            });
        wait_for_treelets();
        return;
    }
    wait_for_treelets();
    if (!climb) return;
    for (int i = p; i < n - 1; i += kTopItems) counter[i] = 0u;
    __syncthreads();
    for (int r = p; r < R; r += kTopItems) climb_range(r, n, prim, tri, nodes, child, parent_int, parent_leaf, counter, cut_a, cut_m);
}
// the same over the whole GPU, with the counters zeroed before it (karras_kernel)
__global__ void __launch_bounds__(256) morton_top_kernel(int n, const uint32_t* prim, const float4* __restrict__ tri, float4* nodes, const int* child,
                                                         const int* parent_int, const int* parent_leaf, uint32_t* counter,
                                                         const uint32_t* __restrict__ cut_a, const uint32_t* __restrict__ cut_m,
                                                         const uint32_t* __restrict__ ncut) {
    const int R = (int)*ncut;
    if (top_by_area(R, n)) return;
    for (int r = blockIdx.x * 256 + threadIdx.x; r < R; r += gridDim.x * 256)
        climb_range(r, n, prim, tri, nodes, child, parent_int, parent_leaf, counter, cut_a, cut_m);
}

// ---- ellipsoidal-connection hierarchy (Sec. 5 "Ellipsoidal Path Connection": nodes weighted by
// the area of the triangles below them).  The implicit binary tree over triangle index ranges
// (GeomDev::enode): eP leaves (a power of two >= nt), node n with children 2n and 2n + 1.
constexpr int kEllBlock = 256;

__device__ __forceinline__ void enode_merge(float4 alo, float4 ahi, float4 blo, float4 bhi, float4& lo, float4& hi) {
    lo = make_float4(fminf(alo.x, blo.x), fminf(alo.y, blo.y), fminf(alo.z, blo.z), alo.w + blo.w);
    hi = make_float4(fmaxf(ahi.x, bhi.x), fmaxf(ahi.y, bhi.y), fmaxf(ahi.z, bhi.z), 0.f);
}

// leaves and the `levels` levels above them, one block per blockDim.x leaves (blockDim.x divides P)
__global__ void __launch_bounds__(kEllBlock) etree_low_kernel(int nt, int P, int levels, const float4* __restrict__ tri,
                                                              float4* __restrict__ node) {
    __shared__ float4 slo[kEllBlock], shi[kEllBlock];
    const int t = threadIdx.x;
    const int i = blockIdx.x * blockDim.x + t;
    float4 lo = make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.f), hi = make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.f);
    if (i < nt) {
        float4 a = tri[3 * (size_t)i], b = tri[3 * (size_t)i + 1], c = tri[3 * (size_t)i + 2];
        float3 v0 = make_float3(a.x, a.y, a.z), e1 = make_float3(b.x, b.y, b.z), e2 = make_float3(c.x, c.y, c.z);
        float3 v1 = make_float3(v0.x + e1.x, v0.y + e1.y, v0.z + e1.z), v2 = make_float3(v0.x + e2.x, v0.y + e2.y, v0.z + e2.z);
        float cx = e1.y * e2.z - e1.z * e2.y, cy = e1.z * e2.x - e1.x * e2.z, cz = e1.x * e2.y - e1.y * e2.x;
        lo = make_float4(fminf(v0.x, fminf(v1.x, v2.x)), fminf(v0.y, fminf(v1.y, v2.y)), fminf(v0.z, fminf(v1.z, v2.z)),
                         0.5f * sqrtf(cx * cx + cy * cy + cz * cz));
        hi = make_float4(fmaxf(v0.x, fmaxf(v1.x, v2.x)), fmaxf(v0.y, fmaxf(v1.y, v2.y)), fmaxf(v0.z, fmaxf(v1.z, v2.z)), 0.f);
    }
    node[2 * (size_t)(P + i)] = lo;
    node[2 * (size_t)(P + i) + 1] = hi;
    slo[t] = lo;
    shi[t] = hi;
    for (int h = 1; h <= levels; ++h) {
        __syncthreads();
        const int cnt = (int)blockDim.x >> h;
        float4 nlo, nhi;
        if (t < cnt) enode_merge(slo[2 * t], shi[2 * t], slo[2 * t + 1], shi[2 * t + 1], nlo, nhi);
        __syncthreads();
        if (t < cnt) {
            slo[t] = nlo;
            shi[t] = nhi;
            const size_t n = (size_t)((P + (int)(blockIdx.x * blockDim.x)) >> h) + t;
            node[2 * n] = nlo;
            node[2 * n + 1] = nhi;
        }
    }
}

// the levels above: nodes [cnt, 2 cnt) for cnt = lowest / 2, ..., 1, one block
__global__ void __launch_bounds__(1024) etree_top_kernel(int lowest, float4* node) {
    for (int cnt = lowest >> 1; cnt >= 1; cnt >>= 1) {
        for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
            const size_t n = (size_t)cnt + t;
            float4 lo, hi;
            enode_merge(node[4 * n], node[4 * n + 1], node[4 * n + 2], node[4 * n + 3], lo, hi);
            node[2 * n] = lo;
            node[2 * n + 1] = hi;
        }
        __syncthreads();
    }
}

// ---- host launchers --------------------------------------------------------------------------
static inline unsigned blocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

cudaError_t launch_xform(int nt, const float* vloc, const uint32_t* tris, const uint32_t* triobj, const uint32_t* objmat,
                         const float* xf, float4* tri_out, float4* cent, uint32_t* bb, cudaStream_t s) {
    note_launch();
    xform_kernel<<<blocks(nt, 256), 256, 0, s>>>(nt, vloc, tris, triobj, objmat, xf, tri_out, cent, bb);
    return cudaGetLastError();
}

// blocks of the cooperative sort (a form of it) that are resident at once, found once per device and process
static int sort_blocks(const void* kernel, int form) {
    static std::atomic<int> known[2][64];   // 1 + the number
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 0;
    int v = known[form][dev].load();
    if (!v) {
        int sms = 0, per = 0, coop = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 256, 0);
        cudaGetLastError();
        v = 1 + (coop ? sms * per : 0);
        known[form][dev].store(v);
    }
    return v - 1;
}
// Which sort, us for n triangles (every block adds up the histograms / rows scanned / separate launches, three a pass):
// 10k 28 / 60 / 60, 40k 39 / 43 / 61, 66k 42 / 41 / 62, 98k 62 / 44 / 62, 198k 93 / 51 / 63, 270k 147 / 58 / 61, 400k 274 / 75 / 65;
// separate 1M 83, 2M 113.  (Tiles of 2048 keys in one launch, as of old for more than 98,304: 198k 82, 400k 130, 1M 268;
// tiles of 1024 with scanned rows: 400k 62, elsewhere slower than the best of these.)
constexpr int kAddTiles = 110, kScanTiles = 600;

// full build of the hierarchy (prim order, children, parents) from the centroids, n > kWhole
cudaError_t launch_build_topology(int n, const float4* cent, uint32_t* bb, uint32_t* keys, uint32_t* vals, uint32_t* keys2,
                                  uint32_t* vals2, int* child, int* parent_int, int* parent_leaf,
                                  uint32_t* counter, uint32_t** prim_out, float4* scratch, cudaStream_t s) {
    note_launch();
    bounds_kernel<<<min(1024u, blocks(n, 256)), 256, 0, s>>>(n, cent, bb);
    note_launch();
    morton_kernel<<<blocks(n, 256), 256, 0, s>>>(n, cent, bb, keys, vals);
    uint32_t *ki = keys, *vi = vals, *ko = keys2, *vo = vals2;
    // the histograms (and the scans' totals) lie in the centroids' memory, which the Morton codes were the last to
    // read: at most 2 B a key and 2 KB of its 16 B a key (n > kWhole)
    uint32_t* counts = reinterpret_cast<uint32_t*>(scratch);
    int nt = (n + kCoopTile - 1) / kCoopTile;
    const void* sort = nt <= kAddTiles ? (const void*)radix_sort_coop_kernel<false> : (const void*)radix_sort_coop_kernel<true>;
    if (nt <= kScanTiles && nt <= sort_blocks(sort, nt <= kAddTiles ? 0 : 1)) {
        int nn = n;
        void* args[] = {&ki, &vi, &ko, &vo, &nn, &counts, &nt};
        note_launch();
        const cudaError_t e = cudaLaunchCooperativeKernel(sort, dim3(nt), dim3(256), args, 0, s);
        if (e != cudaSuccess) return e;
    } else {
        const int ntiles = (n + kTile - 1) / kTile;
        uint32_t* totals = counts + (size_t)256 * ntiles;
        for (int shift = 0; shift < 32; shift += 8) {
            note_launch(3);
            radix_hist_kernel<<<ntiles, 256, 0, s>>>(ki, n, shift, counts, ntiles);
            radix_scan_kernel<<<256, 256, 0, s>>>(counts, totals, ntiles);
            radix_scatter_kernel<<<ntiles, 256, 0, s>>>(ki, vi, ko, vo, n, shift, counts, totals, ntiles);
            uint32_t* t = ki; ki = ko; ko = t;
            t = vi; vi = vo; vo = t;
        }
    }
    // after 4 passes the sorted keys / prims are back in keys / vals
    note_launch();
    karras_kernel<<<blocks(n - 1, 256), 256, 0, s>>>(n, ki, child, parent_int, parent_leaf, keys2, vals2, bb + 6, n > kClimbBlock ? counter : nullptr);
    *prim_out = vi;
    return cudaGetLastError();
}

static cudaError_t size_treelets() {
    static std::atomic<bool> sized[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && sized[dev].load()) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(treelet_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sweep<kTreelet>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(treelet_top_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sweep<kTopItems>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(whole_kernel<kTreelet, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sweep<kTreelet>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(whole_kernel<kWhole, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sweep<kWhole>));
    if (e == cudaSuccess && dev >= 0 && dev < 64) sized[dev].store(true);
    return e;
}

// whether a full build of n triangles is launch_whole's; else launch_build_topology and launch_treelets
bool whole_build(int n) { return n > 1 && n <= kWhole; }
cudaError_t launch_whole(int n, uint32_t* prim, const float4* tri, float4* leaf, float4* nodes, int* child, int* parent_int, int* parent_leaf,
                         cudaStream_t s) {
    const cudaError_t e = size_treelets();
    if (e != cudaSuccess) return e;
    note_launch();
    if (n <= kTreelet)
        whole_kernel<kTreelet, true><<<1, kTreelet, sizeof(Sweep<kTreelet>), s>>>(n, prim, tri, leaf, nodes, child, parent_int, parent_leaf);
    else
        whole_kernel<kWhole, false><<<1, kWhole, sizeof(Sweep<kWhole>), s>>>(n, prim, tri, leaf, nodes, child, parent_int, parent_leaf);
    return cudaGetLastError();
}

// boxes, leaf records and the treelets' topology of a full build, after launch_build_topology
cudaError_t launch_treelets(int n, uint32_t* prim, const float4* tri, float4* leaf, float4* nodes, int* child, int* parent_int,
                            int* parent_leaf, uint32_t* counter, const uint32_t* cut_a, const uint32_t* cut_m, const uint32_t* ncut,
                            float4* boxes, int sms, cudaStream_t s) {
    cudaError_t e = size_treelets();
    if (e != cudaSuccess) return e;
    const bool climb = n > kClimbBlock;   // by a kernel of its own
    // ranges hold at least a few leaves each, mostly hundreds: a block takes several where there are many
    const int grid = min((int)blocks(n, 64), kTreeletBlocks * sms);
    note_launch(3);
    range_box_kernel<<<min((int)blocks(n, 64), 4 * sms), 128, 0, s>>>(n, prim, tri, boxes, cut_a, cut_m, ncut);
    treelet_kernel<<<grid, kTreelet, sizeof(Sweep<kTreelet>), s>>>(n, prim, tri, leaf, nodes, child, parent_int, parent_leaf, cut_a, cut_m, ncut);
    cudaLaunchAttribute beside[1];
    beside[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    beside[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1); cfg.blockDim = dim3(kTopItems); cfg.dynamicSmemBytes = sizeof(Sweep<kTopItems>); cfg.stream = s;
    cfg.attrs = beside; cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, treelet_top_kernel, n, (const uint32_t*)prim, tri, (const float4*)boxes, nodes, child, parent_int,
                           parent_leaf, counter, cut_a, cut_m, ncut, !climb);
    if (e != cudaSuccess) return e;
    if (climb) {
        note_launch();
        morton_top_kernel<<<min((int)blocks(n, 64 * 256), 4 * sms), 256, 0, s>>>(n, prim, tri, nodes, child, parent_int, parent_leaf, counter, cut_a,
                                                                                 cut_m, ncut);
    }
    return cudaGetLastError();
}

cudaError_t launch_refit(int n, const uint32_t* prim, const float4* tri, float4* leaf, float4* nodes, const int* child,
                         const int* parent_int, const int* parent_leaf, uint32_t* counter, cudaStream_t s) {
    if (n > 1) {
        cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(uint32_t) * (size_t)(n - 1), s);
        if (e != cudaSuccess) return e;
    }
    note_launch();
    refit_kernel<<<blocks(n, 256), 256, 0, s>>>(n, prim, tri, leaf, nodes, child, parent_int, parent_leaf, counter);
    return cudaGetLastError();
}

cudaError_t launch_etree(int nt, int P, const float4* tri, float4* node, cudaStream_t s) {
    const int bs = P < kEllBlock ? P : kEllBlock;
    int levels = 0;
    while ((1 << levels) < bs) ++levels;
    note_launch();
    etree_low_kernel<<<P / bs, bs, 0, s>>>(nt, P, levels, tri, node);
    if (P / bs > 1) { note_launch(); etree_top_kernel<<<1, 1024, 0, s>>>(P / bs, node); }
    return cudaGetLastError();
}

}  // namespace tof
