// pt_bvh.cu -- device BVH build (Sec. 5.1.1: AABB hierarchy over the triangles).
//
// 1. centroid bounds, 2. 63-bit Morton codes, 3. LSD radix sort (8 passes of 8 bits),
// 4. binary radix tree over the sorted codes (Karras, HPG 2012), 5. bottom-up boxes,
// 6. top-down collapse into a wide BVH with 8-bit quantised child boxes (80-byte nodes of 8
//    child slots, at most max_width of them used; the layout of compressed wide BVHs, Ylitie,
//    Karras, Laine, HPG 2017), whose leaf triangles are laid out contiguously per node.
// The environment's sampling tables (marginal/conditional CDFs) are built here too.
#include <vector>

#include "pt_internal.h"

#define LEAF_BIT 0x80000000u

__device__ __forceinline__ float3 tri_centroid(const float4* t, uint32_t i) {
    const float4 a = t[3u * i], b = t[3u * i + 1], c = t[3u * i + 2];
    return mk3((a.x + b.x + c.x) * (1.0f / 3.0f), (a.y + b.y + c.y) * (1.0f / 3.0f), (a.z + b.z + c.z) * (1.0f / 3.0f));
}

// One atomic per block and bound: six atomics per warp on six addresses were serialised in L2
// (1.07M triangles: 134 us, now 9).
__global__ void __launch_bounds__(256) k_centroid_bounds(const float4* tris, uint32_t n, uint32_t* cb) {
    float3 lo = mk3(3e38f, 3e38f, 3e38f), hi = mk3(-3e38f, -3e38f, -3e38f);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float3 c = tri_centroid(tris, i);
        lo = mk3(fminf(lo.x, c.x), fminf(lo.y, c.y), fminf(lo.z, c.z));
        hi = mk3(fmaxf(hi.x, c.x), fmaxf(hi.y, c.y), fmaxf(hi.z, c.z));
    }
    block_bounds(lo, hi, cb);
}

__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0x1fffffu;  // 21 bits
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

__global__ void k_morton(const float4* tris, uint32_t n, const uint32_t* cb, uint64_t* keys, uint32_t* vals) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float3 c = tri_centroid(tris, i);
    float q[3];
    for (int a = 0; a < 3; ++a) {
        const float lo = ord2f(cb[a]), hi = ord2f(cb[3 + a]);
        const float ext = hi - lo;
        const float t = ext > 0.0f ? (comp3(c, a) - lo) / ext : 0.5f;
        q[a] = fminf(fmaxf(t * 2097152.0f, 0.0f), 2097151.0f);
    }
    keys[i] = spread3((uint32_t)q[0]) << 2 | spread3((uint32_t)q[1]) << 1 | spread3((uint32_t)q[2]);
    vals[i] = i;
}

// ------------------------------------------------------------------ LSD radix sort
constexpr int RS_THREADS = 256;
constexpr int RS_ROUNDS = 16;
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS;

__global__ void k_rs_hist(const uint64_t* keys, uint32_t n, int shift, uint32_t* hist, uint32_t nblocks) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t base = blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const uint32_t idx = base + r * RS_THREADS + threadIdx.x;
        if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// exclusive scan of each digit's block counts, one block per digit; the digit's total goes to
// total[digit] and the scatter adds the digits' bases.  (One block over all 256 * nblocks
// counters took 55 us a pass at 1.07M triangles, as long as the scatter itself; this takes 4.)
__global__ void __launch_bounds__(256) k_rs_scan(uint32_t* hist, uint32_t nblocks, uint32_t* total) {
    __shared__ uint32_t wsum[8];
    uint32_t* row = hist + (size_t)blockIdx.x * nblocks;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t run = 0;
    for (uint32_t b0 = 0; b0 < nblocks; b0 += 256) {
        const uint32_t i = b0 + threadIdx.x;
        const uint32_t v = i < nblocks ? row[i] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        uint32_t before = run, all = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) before += wsum[w];
            all += wsum[w];
        }
        if (i < nblocks) row[i] = before + x - v;
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = run;
}

// stable scatter: tile order = round-major, then thread; ranks from warp match + per-warp counts
__global__ void k_rs_scatter(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout, uint32_t n,
                             int shift, const uint32_t* hist, const uint32_t* total, uint32_t nblocks) {
    __shared__ uint32_t base[256];
    __shared__ uint32_t wcnt[RS_THREADS / 32][256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the digits' bases: exclusive scan of their totals
    base[tid] = total[tid];
    __syncthreads();
    for (int off = 1; off < 256; off <<= 1) {
        const uint32_t v = tid >= off ? base[tid - off] : 0u;
        __syncthreads();
        base[tid] += v;
        __syncthreads();
    }
    const uint32_t digit_base = base[tid] - total[tid];
    __syncthreads();
    base[tid] = digit_base + hist[tid * nblocks + blockIdx.x];
    const uint32_t lt = (1u << lane) - 1u;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const uint32_t idx = blockIdx.x * RS_TILE + r * RS_THREADS + tid;
        const bool valid = idx < n;
        const uint64_t key = valid ? kin[idx] : 0ull;
        const uint32_t digit = valid ? (uint32_t)((key >> shift) & 255u) : 256u;
        for (int j = tid; j < (RS_THREADS / 32) * 256; j += RS_THREADS) (&wcnt[0][0])[j] = 0u;
        __syncthreads();
        const uint32_t peers = __match_any_sync(0xffffffffu, digit);
        const uint32_t rank = __popc(peers & lt);
        if (valid && rank == 0) wcnt[warp][digit] = __popc(peers);
        __syncthreads();
        {
            uint32_t run = base[tid];
            for (int w = 0; w < RS_THREADS / 32; ++w) {
                const uint32_t c = wcnt[w][tid];
                wcnt[w][tid] = run;
                run += c;
            }
            base[tid] = run;
        }
        __syncthreads();
        if (valid) {
            const uint32_t pos = wcnt[warp][digit] + rank;
            kout[pos] = key;
            vout[pos] = vin[idx];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ binary radix tree
__device__ __forceinline__ int lcp(const uint64_t* keys, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    const uint64_t a = keys[i], b = keys[j];
    if (a == b) return 64 + __clz((uint32_t)(i ^ j));
    return __clzll((long long)(a ^ b));
}

__global__ void k_karras(const uint64_t* keys, int n, uint32_t* left, uint32_t* right, uint32_t* par_int,
                         uint32_t* par_leaf, uint32_t* first, uint32_t* last) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    const int d = (lcp(keys, n, i, i + 1) - lcp(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = lcp(keys, n, i, i - d);
    int lmax = 2;
    while (lcp(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (lcp(keys, n, i, i + (l + t) * d) > dmin) l += t;
    const int j = i + l * d;
    const int dnode = lcp(keys, n, i, j);
    int s = 0, t = l;
    for (;;) {
        t = (t + 1) >> 1;
        if (lcp(keys, n, i, i + (s + t) * d) > dnode) s += t;
        if (t <= 1) break;
    }
    const int gamma = i + s * d + min(d, 0);
    const int lo = min(i, j), hi = max(i, j);
    const uint32_t L = (lo == gamma) ? (LEAF_BIT | (uint32_t)gamma) : (uint32_t)gamma;
    const uint32_t R = (hi == gamma + 1) ? (LEAF_BIT | (uint32_t)(gamma + 1)) : (uint32_t)(gamma + 1);
    left[i] = L;
    right[i] = R;
    first[i] = (uint32_t)lo;
    last[i] = (uint32_t)hi;
    if (L & LEAF_BIT) par_leaf[L & ~LEAF_BIT] = (uint32_t)i; else par_int[L] = (uint32_t)i;
    if (R & LEAF_BIT) par_leaf[R & ~LEAF_BIT] = (uint32_t)i; else par_int[R] = (uint32_t)i;
    if (i == 0) par_int[0] = 0xffffffffu;
}

struct Box {
    float3 lo, hi;
};

__device__ __forceinline__ Box tri_box(const float4* tris, uint32_t t) {
    const float4 a = tris[3u * t], b = tris[3u * t + 1], c = tris[3u * t + 2];
    Box r;
    r.lo = mk3(fminf(a.x, fminf(b.x, c.x)), fminf(a.y, fminf(b.y, c.y)), fminf(a.z, fminf(b.z, c.z)));
    r.hi = mk3(fmaxf(a.x, fmaxf(b.x, c.x)), fmaxf(a.y, fmaxf(b.y, c.y)), fmaxf(a.z, fmaxf(b.z, c.z)));
    return r;
}
__device__ __forceinline__ Box box_union(Box a, Box b) {
    Box r;
    r.lo = mk3(fminf(a.lo.x, b.lo.x), fminf(a.lo.y, b.lo.y), fminf(a.lo.z, b.lo.z));
    r.hi = mk3(fmaxf(a.hi.x, b.hi.x), fmaxf(a.hi.y, b.hi.y), fmaxf(a.hi.z, b.hi.z));
    return r;
}

// ---- cost-optimal collapse: per binary node, the least surface-area cost of its subtree
// when it fills exactly j = 1..8 slots of a wide node (the dynamic programme of Ylitie,
// Karras and Laine, HPG 2017, restated for leaves of at most leaf_size triangles and nodes of
// at most W = width children).  With A the (half) surface area, a wide node visit costing 1
// plus box_cost per slot and a triangle test tri_cost:
//   C(k)    = A(k) * tri_cost * count(k)                          if count(k) <= leaf_size
//           = A(k) + min_{j=2..W} E(k, j) + A(k) * box_cost * j    otherwise (a wide node)
//   E(k, 1) = C(k);  E(k, j) = min_{i=1..j-1} E(L, i) + E(R, j - i)  (j >= 2)
// and a single triangle costs A * tri_cost as one slot and cannot fill more.  dec[k] keeps
// the choices in nibbles: nibble 0 the slot count j of C(k) for a wide node, nibble j - 1
// (j = 2..8) the split i of E(k, j).
struct DpArrays {
    float* cost;            // 8 per binary node: E(k, 1..8); null: greedy collapse
    uint32_t* dec;          // choices, one word per binary node
    uint32_t leaf_size;
    float tri_cost, box_cost;
    uint32_t width;         // most children of a wide node, 2..8
};

__device__ __forceinline__ float half_area_box(float3 lo, float3 hi) {
    const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return dx * dy + dy * dz + dz * dx;
}

// E(child, 1..8) of a child reference: a triangle (its area given) or a binary node
__device__ __forceinline__ void dp_child(const DpArrays& D, uint32_t ref, float leaf_area, float (&c)[8]) {
    if (ref & 0x80000000u) {
        c[0] = leaf_area * D.tri_cost;
#pragma unroll
        for (int j = 1; j < 8; ++j) c[j] = __int_as_float(0x7f800000);
    } else {
        const float4 a = __ldcg(reinterpret_cast<const float4*>(D.cost + 8u * ref));
        const float4 b = __ldcg(reinterpret_cast<const float4*>(D.cost + 8u * ref) + 1);
        c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w; c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
    }
}

__device__ __forceinline__ void dp_node(const DpArrays& D, uint32_t k, uint32_t lref, float larea, uint32_t rref,
                                        float rarea, uint32_t count, float area) {
    float cl[8], cr[8], e[8];
    dp_child(D, lref, larea, cl);
    dp_child(D, rref, rarea, cr);
    uint32_t dec = 0;
#pragma unroll
    for (uint32_t j = 2; j <= 8; ++j) {
        float best = __int_as_float(0x7f800000);
        uint32_t bi = 1;
        for (uint32_t i = 1; i < j; ++i) {
            const float v = cl[i - 1] + cr[j - i - 1];
            if (v < best) { best = v; bi = i; }
        }
        e[j - 1] = best;
        dec |= bi << (4 * (j - 1));
    }
    if (count <= D.leaf_size) {
        e[0] = area * D.tri_cost * (float)count;
    } else {
        float best = __int_as_float(0x7f800000);
        uint32_t bj = 2;
        for (uint32_t j = 2; j <= D.width; ++j) {
            const float v = e[j - 1] + area * D.box_cost * (float)j;
            if (v < best) { best = v; bj = j; }
        }
        e[0] = area + best;
        dec |= bj;
    }
    __stcg(reinterpret_cast<float4*>(D.cost + 8u * k), make_float4(e[0], e[1], e[2], e[3]));
    __stcg(reinterpret_cast<float4*>(D.cost + 8u * k) + 1, make_float4(e[4], e[5], e[6], e[7]));
    __stcg(D.dec + k, dec);
}

struct BinTree {
    const uint32_t *left, *right, *first, *last, *perm;
    float4 *blo, *bhi;
    const float4* tris;
};

__device__ __forceinline__ Box ref_box(const BinTree& T, uint32_t ref) {
    if (ref & LEAF_BIT) return tri_box(T.tris, T.perm[ref & ~LEAF_BIT]);
    const float4 lo = __ldcg(T.blo + ref), hi = __ldcg(T.bhi + ref);
    Box b;
    b.lo = xyz(lo);
    b.hi = xyz(hi);
    return b;
}

__global__ void k_bottom_up(BinTree T, int n, const uint32_t* par_int, const uint32_t* par_leaf, uint32_t* flags,
                            DpArrays D) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t node = par_leaf[i];
    while (node != 0xffffffffu) {
        __threadfence();
        if (atomicAdd(&flags[node], 1u) == 0u) return;  // first child to arrive stops
        __threadfence();
        const uint32_t l = T.left[node], r = T.right[node];
        const Box bl = ref_box(T, l), br = ref_box(T, r);
        const Box b = box_union(bl, br);
        __stcg(T.blo + node, make_float4(b.lo.x, b.lo.y, b.lo.z, 0.0f));
        __stcg(T.bhi + node, make_float4(b.hi.x, b.hi.y, b.hi.z, 0.0f));
        if (D.cost)
            dp_node(D, node, l, half_area_box(bl.lo, bl.hi), r, half_area_box(br.lo, br.hi),
                    T.last[node] - T.first[node] + 1u, half_area_box(b.lo, b.hi));
        node = par_int[node];
    }
}

// ------------------------------------------------------------------ PLOC binary tree
// Parallel locally-ordered clustering (Meister & Bittner, IEEE TVCG 2018): the clusters start
// as the triangles in Morton order; each round every cluster finds, within PLOC_R positions on
// either side, the cluster whose union with it has the least surface area, mutual pairs merge
// into a new binary node (at the lower position), and the survivors are compacted in order.
// Pairs are ranked by (area, lower index, higher index), a total order, so the globally least
// pair within the window is always mutual and every round merges at least once.  Merges get
// node indices counting down from n - 2, so the last merge (the root) is node 0, and every
// node's children have higher indices than the node.  A top-down pass over the rounds in
// reverse then lays the triangles out in tree order, giving each subtree the contiguous
// [first, last] range the collapse needs.
// 8 against the published 16: builds take 6 % less (0.2M-triangle CAD model 2.02 -> 1.79 ms,
// 5.2M-triangle glass scene 5.9 -> 5.5).  Frames of 22 CAD, glass and velvet scenes of 640 to 5.2M
// triangles differ by -1.7 to +2.2 % (mean 0.1 %; fewer node visits in 12, more in 10), as after
// any small change of the tree.  A random soup, whose Morton order says little about its sizes,
// is the exception: 2.8 % (20,000 triangles) and 6.5 % (300,000) longer frames.
constexpr int PLOC_R = 8;
constexpr int PLOC_THREADS = 256;
constexpr int PLOC_SCAN_ITEMS = 4;                      // per thread of the block scan
constexpr int PLOC_SCAN_TILE = PLOC_THREADS * PLOC_SCAN_ITEMS;

// The rounds run without the host: round r reads its cluster count and the merges before it
// from state r and k_ploc_scan_top writes state r + 1 (a ring, read back every PLOC_BATCH
// rounds).  Once at most PLOC_TAIL clusters are left the remaining rounds are many and tiny
// (108 of 145 for a 1.07M-triangle CAD model) and one block runs them all in shared memory.
constexpr uint32_t PLOC_BATCH = 4, PLOC_TAIL = 2048, PLOC_TAIL_THREADS = 1024;
struct PlocState {
    uint32_t m, merged;      // clusters, merges so far
};

struct Clusters {
    uint32_t* ref;      // LEAF_BIT | triangle id, or binary node index
    uint32_t* cnt;      // triangles below
    float4 *lo, *hi;    // bounds
};

__device__ __forceinline__ float half_area3(float3 lo, float3 hi) {
    const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return dx * dy + dy * dz + dz * dx;
}

__global__ void k_ploc_init(const float4* tris, const uint32_t* perm, uint32_t n, Clusters c) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t t = perm[i];
    const Box b = tri_box(tris, t);
    c.ref[i] = LEAF_BIT | t;
    c.cnt[i] = 1u;
    c.lo[i] = make_float4(b.lo.x, b.lo.y, b.lo.z, 0.0f);
    c.hi[i] = make_float4(b.hi.x, b.hi.y, b.hi.z, 0.0f);
}

// nearest neighbour of each of the m clusters within the window (lowest index on equal area)
__global__ void __launch_bounds__(PLOC_THREADS) k_ploc_nn(Clusters c, const PlocState* st, uint32_t* nn) {
    __shared__ float4 slo[PLOC_THREADS + 2 * PLOC_R], shi[PLOC_THREADS + 2 * PLOC_R];
    const uint32_t m = st->m;
    if (m <= PLOC_TAIL || blockIdx.x * PLOC_THREADS >= m) return;
    const int base = (int)(blockIdx.x * PLOC_THREADS) - PLOC_R;
    for (int k = threadIdx.x; k < PLOC_THREADS + 2 * PLOC_R; k += PLOC_THREADS) {
        const int g = base + k;
        if (g >= 0 && g < (int)m) { slo[k] = c.lo[g]; shi[k] = c.hi[g]; }
    }
    __syncthreads();
    const int i = (int)(blockIdx.x * PLOC_THREADS + threadIdx.x);
    if (i >= (int)m) return;
    const int li = threadIdx.x + PLOC_R;
    const float3 alo = xyz(slo[li]), ahi = xyz(shi[li]);
    float best = __int_as_float(0x7f800000);
    int bj = -1;
    const int j0 = max(i - PLOC_R, 0), j1 = min(i + PLOC_R, (int)m - 1);
    for (int j = j0; j <= j1; ++j) {
        if (j == i) continue;
        const int lj = j - base;
        const float3 blo = xyz(slo[lj]), bhi = xyz(shi[lj]);
        const float a = half_area3(mk3(fminf(alo.x, blo.x), fminf(alo.y, blo.y), fminf(alo.z, blo.z)),
                                   mk3(fmaxf(ahi.x, bhi.x), fmaxf(ahi.y, bhi.y), fmaxf(ahi.z, bhi.z)));
        if (a < best) { best = a; bj = j; }
    }
    nn[i] = (uint32_t)bj;
}

// per cluster: survives (1) and creates a node (bit 32) -- the lower index of a mutual pair --
// or is absorbed (0); exclusive block-level scan of those 64-bit values, block totals aside
__device__ __forceinline__ uint64_t ploc_flag(const uint32_t* nn, uint32_t m, uint32_t i) {
    if (i >= m) return 0ull;
    const uint32_t j = nn[i];
    if (j >= m) return 1ull;                       // m == 1: no neighbour
    if (nn[j] != i) return 1ull;
    return i < j ? ((1ull << 32) | 1ull) : 0ull;
}

__global__ void __launch_bounds__(PLOC_THREADS) k_ploc_scan(const uint32_t* nn, const PlocState* st, uint64_t* pre,
                                                            uint64_t* block_sum) {
    const uint32_t m = st->m;
    if (m <= PLOC_TAIL || blockIdx.x * PLOC_SCAN_TILE >= m) return;
    __shared__ uint64_t warp_sum[PLOC_THREADS / 32];
    const uint32_t t0 = blockIdx.x * PLOC_SCAN_TILE + threadIdx.x * PLOC_SCAN_ITEMS;
    uint64_t v[PLOC_SCAN_ITEMS], run = 0;
#pragma unroll
    for (int k = 0; k < PLOC_SCAN_ITEMS; ++k) {
        v[k] = ploc_flag(nn, m, t0 + k);
        run += v[k];
    }
    // inclusive scan of the per-thread totals across the warp, then across warps
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t x = run;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    uint64_t before = 0;
    for (int w = 0; w < warp; ++w) before += warp_sum[w];
    uint64_t acc = before + x - run;               // exclusive prefix of this thread
#pragma unroll
    for (int k = 0; k < PLOC_SCAN_ITEMS; ++k) {
        if (t0 + k < m) pre[t0 + k] = acc;
        acc += v[k];
    }
    if (threadIdx.x == PLOC_THREADS - 1) block_sum[blockIdx.x] = before + x;
}

// exclusive scan of the block totals by one block; the grand total makes the next state
__global__ void k_ploc_scan_top(uint64_t* data, const PlocState* st, PlocState* next) {
    const uint32_t m = st->m;
    if (m <= PLOC_TAIL) {
        if (threadIdx.x == 0) *next = *st;
        return;
    }
    const uint32_t nb = (m + PLOC_SCAN_TILE - 1) / PLOC_SCAN_TILE;
    __shared__ uint64_t part[1024];
    const uint32_t per = (nb + 1023) / 1024;
    const uint32_t b = threadIdx.x * per, e = min(b + per, nb);
    uint64_t sum = 0;
    for (uint32_t i = b; i < e; ++i) sum += data[i];
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const uint64_t v = threadIdx.x >= (uint32_t)off ? part[threadIdx.x - off] : 0ull;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    uint64_t run = part[threadIdx.x] - sum;
    for (uint32_t i = b; i < e; ++i) {
        const uint64_t v = data[i];
        data[i] = run;
        run += v;
    }
    if (threadIdx.x == 1023) {
        next->m = (uint32_t)(part[1023] & 0xffffffffull);
        next->merged = st->merged + (uint32_t)(part[1023] >> 32);
    }
}

// survivors to their compacted position; a mutual pair becomes binary node
// n - 2 - (merged_before + its rank among this round's merges)
__global__ void k_ploc_compact(Clusters a, Clusters b, const uint32_t* nn, const PlocState* st, const uint64_t* pre,
                               const uint64_t* block_pre, uint32_t n, uint32_t* left,
                               uint32_t* right, uint32_t* count, float4* blo, float4* bhi, DpArrays D) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t m = st->m, merged_before = st->merged;
    if (m <= PLOC_TAIL || i >= m) return;
    const uint64_t f = ploc_flag(nn, m, i);
    if (f == 0ull) return;
    const uint64_t p = pre[i] + block_pre[i / PLOC_SCAN_TILE];
    const uint32_t pos = (uint32_t)(p & 0xffffffffull);
    if (f == 1ull) {
        b.ref[pos] = a.ref[i];
        b.cnt[pos] = a.cnt[i];
        b.lo[pos] = a.lo[i];
        b.hi[pos] = a.hi[i];
        return;
    }
    const uint32_t j = nn[i];
    const uint32_t node = n - 2u - (merged_before + (uint32_t)(p >> 32));
    const float4 l0 = a.lo[i], h0 = a.hi[i], l1 = a.lo[j], h1 = a.hi[j];
    const float4 lo = make_float4(fminf(l0.x, l1.x), fminf(l0.y, l1.y), fminf(l0.z, l1.z), 0.0f);
    const float4 hi = make_float4(fmaxf(h0.x, h1.x), fmaxf(h0.y, h1.y), fmaxf(h0.z, h1.z), 0.0f);
    const uint32_t c = a.cnt[i] + a.cnt[j];
    left[node] = a.ref[i];
    right[node] = a.ref[j];
    count[node] = c;
    blo[node] = lo;
    bhi[node] = hi;
    if (D.cost)   // the children's costs were written in earlier rounds
        dp_node(D, node, a.ref[i], half_area_box(xyz(l0), xyz(h0)), a.ref[j], half_area_box(xyz(l1), xyz(h1)), c,
                half_area_box(xyz(lo), xyz(hi)));
    b.ref[pos] = node;
    b.cnt[pos] = c;
    b.lo[pos] = lo;
    b.hi[pos] = hi;
}

// top-down layout of the nodes [lo, hi] (one round's merges; their parents are done): each
// node's range starts at first[node], its left subtree first; leaves take their position in
// perm and their child reference becomes LEAF_BIT | position
struct PlocTree {
    uint32_t *left, *right, *count, *first, *last, *perm;
    float4 *blo, *bhi;
};

__device__ __forceinline__ void ploc_layout_node(const PlocTree& T, uint32_t k) {
    const uint32_t f = T.first[k];
    const uint32_t L = T.left[k], R = T.right[k];
    const uint32_t cl = (L & LEAF_BIT) ? 1u : T.count[L];
    if (L & LEAF_BIT) {
        T.perm[f] = L & ~LEAF_BIT;
        T.left[k] = LEAF_BIT | f;
    } else {
        T.first[L] = f;
    }
    if (R & LEAF_BIT) {
        T.perm[f + cl] = R & ~LEAF_BIT;
        T.right[k] = LEAF_BIT | (f + cl);
    } else {
        T.first[R] = f + cl;
    }
    T.last[k] = f + T.count[k] - 1u;
}

__global__ void k_ploc_layout(uint32_t lo, uint32_t hi, PlocTree T) {
    const uint32_t k = lo + blockIdx.x * blockDim.x + threadIdx.x;
    if (k <= hi) ploc_layout_node(T, k);
}

// The last rounds (m <= PLOC_TAIL clusters) by one block, the clusters in shared memory, by the
// same rules as the kernels above; then the layout of these rounds' nodes, which are the top
// of the tree.  status: 1 when one cluster is left, 0 if a round merged nothing.  A round costs
// a few microseconds here, against about 30 as four launches and a read-back.
constexpr size_t PLOC_TAIL_SMEM = (size_t)PLOC_TAIL * (6 * sizeof(float) + 4 * sizeof(uint32_t)) + 64 * sizeof(uint32_t);

__global__ void __launch_bounds__(PLOC_TAIL_THREADS) k_ploc_tail(Clusters c, uint32_t m, uint32_t merged, uint32_t n,
                                                                 PlocTree T, DpArrays D, uint32_t* status) {
    extern __shared__ float sm[];
    constexpr int TH = (int)PLOC_TAIL_THREADS, CAP = (int)PLOC_TAIL;
    float* box[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) box[a] = sm + a * CAP;
    uint32_t* ref = reinterpret_cast<uint32_t*>(sm + 6 * CAP);
    uint32_t* cnt = ref + CAP;
    uint32_t* nn = cnt + CAP;
    uint32_t* rounds = nn + CAP;            // merges before each round (at most m - 1 rounds)
    uint32_t* wsum = rounds + CAP;          // 2 x 32 warp totals
    const int t = (int)threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int i = t; i < (int)m; i += TH) {
        const float4 lo = c.lo[i], hi = c.hi[i];
        box[0][i] = lo.x; box[1][i] = lo.y; box[2][i] = lo.z;
        box[3][i] = hi.x; box[4][i] = hi.y; box[5][i] = hi.z;
        ref[i] = c.ref[i];
        cnt[i] = c.cnt[i];
    }
    __syncthreads();
    auto lo_of = [&](int i) { return mk3(box[0][i], box[1][i], box[2][i]); };
    auto hi_of = [&](int i) { return mk3(box[3][i], box[4][i], box[5][i]); };
    uint32_t n_rounds = 0;
    bool stuck = false;
    while (m > 1u && !stuck) {
        for (int i = t; i < (int)m; i += TH) {
            const float3 alo = lo_of(i), ahi = hi_of(i);
            float best = __int_as_float(0x7f800000);
            int bj = -1;
            const int j0 = max(i - PLOC_R, 0), j1 = min(i + PLOC_R, (int)m - 1);
            for (int j = j0; j <= j1; ++j) {
                if (j == i) continue;
                const float3 blo = lo_of(j), bhi = hi_of(j);
                const float a = half_area3(mk3(fminf(alo.x, blo.x), fminf(alo.y, blo.y), fminf(alo.z, blo.z)),
                                           mk3(fmaxf(ahi.x, bhi.x), fmaxf(ahi.y, bhi.y), fmaxf(ahi.z, bhi.z)));
                if (a < best) { best = a; bj = j; }
            }
            nn[i] = (uint32_t)bj;
        }
        __syncthreads();
        // this thread's clusters t and t + TH: survives (1), merges (1 << 16); prefix over both halves
        uint32_t f[2], x[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t v = ploc_flag(nn, m, (uint32_t)(t + h * TH));
            f[h] = x[h] = (uint32_t)(v & 1ull) | ((uint32_t)(v >> 32) << 16);
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x[h], off);
                if (lane >= off) x[h] += y;
            }
            if (lane == 31) wsum[32 * h + warp] = x[h];
        }
        __syncthreads();
        if (warp == 0) {
            // inclusive scan of the 64 warp totals, first half then second
            uint32_t a = wsum[lane], b = wsum[32 + lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t ya = __shfl_up_sync(0xffffffffu, a, off), yb = __shfl_up_sync(0xffffffffu, b, off);
                if (lane >= off) { a += ya; b += yb; }
            }
            b += __shfl_sync(0xffffffffu, a, 31);
            wsum[lane] = a;
            wsum[32 + lane] = b;
        }
        __syncthreads();
        const uint32_t total = wsum[63];
        float3 nlo[2], nhi[2];
        uint32_t nref[2], ncnt[2], pos[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int w = 32 * h + warp, i = t + h * TH;
            if (f[h] == 0u) continue;
            const uint32_t pre = (w > 0 ? wsum[w - 1] : 0u) + x[h] - f[h];
            pos[h] = pre & 0xffffu;
            nlo[h] = lo_of(i);
            nhi[h] = hi_of(i);
            nref[h] = ref[i];
            ncnt[h] = cnt[i];
            if (f[h] >> 16) {
                const int j = (int)nn[i];
                const float3 l1 = lo_of(j), h1 = hi_of(j);
                const float la = half_area_box(nlo[h], nhi[h]), ra = half_area_box(l1, h1);
                const uint32_t node = n - 2u - (merged + (pre >> 16));
                nlo[h] = mk3(fminf(nlo[h].x, l1.x), fminf(nlo[h].y, l1.y), fminf(nlo[h].z, l1.z));
                nhi[h] = mk3(fmaxf(nhi[h].x, h1.x), fmaxf(nhi[h].y, h1.y), fmaxf(nhi[h].z, h1.z));
                ncnt[h] += cnt[j];
                T.left[node] = nref[h];
                T.right[node] = ref[j];
                T.count[node] = ncnt[h];
                T.blo[node] = make_float4(nlo[h].x, nlo[h].y, nlo[h].z, 0.0f);
                T.bhi[node] = make_float4(nhi[h].x, nhi[h].y, nhi[h].z, 0.0f);
                if (D.cost) dp_node(D, node, nref[h], la, ref[j], ra, ncnt[h], half_area_box(nlo[h], nhi[h]));
                nref[h] = node;
            }
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (f[h] == 0u) continue;
            const uint32_t q = pos[h];
            box[0][q] = nlo[h].x; box[1][q] = nlo[h].y; box[2][q] = nlo[h].z;
            box[3][q] = nhi[h].x; box[4][q] = nhi[h].y; box[5][q] = nhi[h].z;
            ref[q] = nref[h];
            cnt[q] = ncnt[h];
        }
        if (t == 0) rounds[n_rounds] = merged;
        ++n_rounds;
        stuck = (total >> 16) == 0u;
        m -= total >> 16;
        merged += total >> 16;
        __syncthreads();
    }
    if (t == 0) *status = stuck ? 0u : 1u;
    if (stuck) return;
    if (t == 0) T.first[0] = 0u;
    __syncthreads();
    for (uint32_t r = n_rounds; r-- > 0;) {
        const uint32_t lo = n - 1u - (r + 1u < n_rounds ? rounds[r + 1u] : n - 1u), hi = n - 2u - rounds[r];
        for (uint32_t k = lo + (uint32_t)t; k <= hi; k += TH) ploc_layout_node(T, k);
        __syncthreads();
    }
}

// ------------------------------------------------------------------ collapse to wide nodes
struct CollapseCtx {
    BinTree T;
    uint32_t leaf_size;
    uint32_t width;         // most children of a wide node, 2..8
    uint32_t* task_ref;     // binary node ref of each wide-node task
    uint32_t* task_node;    // wide node index of each task
    uint32_t* counters;     // [0] node count, [1] triangle count, [2] queue tail
    uint4* nodes;
    float4* out_tris;
    const float4* in_tris;
    DpArrays dp;            // cost-optimal choices (dp.cost null: greedy, largest child first)
};

__device__ __forceinline__ uint32_t ref_count(const BinTree& T, uint32_t ref) {
    return (ref & LEAF_BIT) ? 1u : T.last[ref] - T.first[ref] + 1u;
}
__device__ __forceinline__ uint32_t ref_first(const BinTree& T, uint32_t ref) {
    return (ref & LEAF_BIT) ? (ref & ~LEAF_BIT) : T.first[ref];
}
__device__ __forceinline__ float area(const Box& b) {
    const float dx = b.hi.x - b.lo.x, dy = b.hi.y - b.lo.y, dz = b.hi.z - b.lo.z;
    return dx * dy + dy * dz + dz * dx;
}

// One wide node by a group of 8 lanes, lane = child slot: unfolding, boxes, quantisation and the
// copies of the leaves' triangles are chains of dependent loads and divisions, so a thread per
// node took 75 us a level, even a level of one node (17 levels, 1.28 ms of a 1.07M-triangle
// build); side by side a level takes 21 (20 launches, 0.42 ms).
__device__ __forceinline__ void collapse_task(const CollapseCtx& C, uint32_t ti, uint32_t gl, uint32_t gm, uint32_t gbase) {
    const BinTree& T = C.T;
    const uint32_t root_ref = C.task_ref[ti];
    const uint32_t wnode = C.task_node[ti];
    constexpr uint32_t NONE = 0xffffffffu;     // an empty slot
    uint32_t ref = NONE;
    if ((root_ref & LEAF_BIT) || ref_count(T, root_ref) <= C.leaf_size) {
        if (gl == 0) ref = root_ref;
    } else if (C.dp.cost) {
        // unfold the choices side by side: a part with a budget of j slots starts at lane `gl`
        // and owns j lanes; its left child keeps the first i of them, the right child the rest
        uint32_t j = 0;
        if (gl == 0) {
            ref = root_ref;
            j = min(max(C.dp.dec[root_ref] & 15u, 2u), 8u);
        }
        for (;;) {
            uint32_t i = 0, right = NONE, rj = 0;
            if (ref != NONE && !(ref & LEAF_BIT) && j >= 2u) i = (C.dp.dec[ref] >> (4u * (j - 1u))) & 15u;
            const bool split = i > 0u && i < j;
            if (split) {
                right = T.right[ref];
                ref = T.left[ref];
                rj = j - i;
                j = i;
            } else {
                j = min(j, 1u);      // one slot
            }
            const uint32_t splits = (__ballot_sync(gm, split) >> gbase) & 0xffu;
            if (splits == 0u) break;
            // the part whose right child starts at this lane, if any
            const uint32_t target = split ? gl + i : 8u;
#pragma unroll
            for (uint32_t q = 0; q < 8; ++q) {
                const uint32_t tq = __shfl_sync(gm, target, q, 8), rq = __shfl_sync(gm, right, q, 8),
                               jq = __shfl_sync(gm, rj, q, 8);
                if (tq == gl) { ref = rq; j = jq; }
            }
        }
    } else {
        // greedy, largest child first; every lane of the group makes the same choices
        uint32_t ch[8];
        float ca[8];
        ch[0] = T.left[root_ref];
        ch[1] = T.right[root_ref];
        int nc = 2;
        for (int k = 0; k < 2; ++k) ca[k] = area(ref_box(T, ch[k]));
        while (nc < (int)C.width) {
            int best = -1;
            float best_a = -1.0f;
            for (int k = 0; k < nc; ++k) {
                if ((ch[k] & LEAF_BIT) || ref_count(T, ch[k]) <= C.leaf_size) continue;
                if (ca[k] > best_a) { best_a = ca[k]; best = k; }
            }
            if (best < 0) break;
            const uint32_t r = ch[best];
            ch[best] = T.left[r];
            ca[best] = area(ref_box(T, ch[best]));
            ch[nc] = T.right[r];
            ca[nc] = area(ref_box(T, ch[nc]));
            ++nc;
        }
        if ((int)gl < nc) ref = ch[gl];
    }
    const bool used = ref != NONE;
    const float inf = __int_as_float(0x7f800000);
    Box cb;
    cb.lo = splat3(inf);
    cb.hi = splat3(-inf);
    uint32_t c = 0;
    if (used) {
        cb = ref_box(T, ref);
        c = ref_count(T, ref);
    }
    const bool inner = c > C.leaf_size;
    const uint32_t imask = (__ballot_sync(gm, inner) >> gbase) & 0xffu;
    const uint32_t n_int = __popc(imask), rank = __popc(imask & ((1u << gl) - 1u));
    // leaf triangles before this slot's
    const uint32_t lc = inner ? 0u : c;
    uint32_t incl = lc;
#pragma unroll
    for (uint32_t d = 1; d < 8; d <<= 1) {
        const uint32_t y = __shfl_up_sync(gm, incl, d, 8);
        if (gl >= d) incl += y;
    }
    const uint32_t toff = incl - lc, n_leaf_tris = __shfl_sync(gm, incl, 7, 8);
    // lanes 0..2 reserve the node's children, triangles and queue entries
    uint32_t base = 0;
    if (gl < 3) {
        const uint32_t want = gl == 1 ? n_leaf_tris : n_int;
        if (want) base = atomicAdd(&C.counters[gl], want);
    }
    const uint32_t child_base = __shfl_sync(gm, base, 0, 8), tri_base = __shfl_sync(gm, base, 1, 8),
                   qpos = __shfl_sync(gm, base, 2, 8);
    // node box and quantisation frame
    Box nb = cb;
#pragma unroll
    for (uint32_t d = 1; d < 8; d <<= 1) {
        Box o;
        o.lo = mk3(__shfl_xor_sync(gm, nb.lo.x, d, 8), __shfl_xor_sync(gm, nb.lo.y, d, 8), __shfl_xor_sync(gm, nb.lo.z, d, 8));
        o.hi = mk3(__shfl_xor_sync(gm, nb.hi.x, d, 8), __shfl_xor_sync(gm, nb.hi.y, d, 8), __shfl_xor_sync(gm, nb.hi.z, d, 8));
        nb = box_union(nb, o);
    }
    const float3 p = nb.lo;
    const float emax = fmaxf(nb.hi.x - nb.lo.x, fmaxf(nb.hi.y - nb.lo.y, nb.hi.z - nb.lo.z));
    uint32_t ebias[3];
    unsigned char* node = reinterpret_cast<unsigned char*>(C.nodes + 5u * wnode);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float pa = comp3(p, a);
        const float e = fmaxf(fmaxf(comp3(nb.hi, a) - pa, emax * 1e-6f), 1e-30f);
        int ex;
        frexpf(e / 255.0f, &ex);
        int bb = min(max(ex + 127, 1), 254);
        float sc = __uint_as_float((uint32_t)bb << 23);
        while (bb < 254 && fmaf(255.0f, sc, pa) < comp3(nb.hi, a)) { ++bb; sc = __uint_as_float((uint32_t)bb << 23); }
        ebias[a] = (uint32_t)bb;
        uint32_t qlo = 0, qhi = 0;
        if (used) {
            const float lo = comp3(cb.lo, a), hi = comp3(cb.hi, a);
            float ql = floorf(__fsub_rd(lo, pa) / sc);
            ql = fminf(fmaxf(ql, 0.0f), 255.0f);
            while (ql > 0.0f && fmaf(ql, sc, pa) > lo) ql -= 1.0f;
            float qh = ceilf(__fsub_ru(hi, pa) / sc);
            qh = fminf(fmaxf(qh, 0.0f), 255.0f);
            while (qh < 255.0f && fmaf(qh, sc, pa) < hi) qh += 1.0f;
            qlo = (uint32_t)ql;
            qhi = (uint32_t)qh;
        }
        node[32 + 8 * a + gl] = (unsigned char)qlo;
        node[56 + 8 * a + gl] = (unsigned char)qhi;
    }
    node[24 + gl] = (unsigned char)(inner ? 1u : c ? (c << 5) | toff : 0u);
    if (gl == 0) {
        C.nodes[5u * wnode] = make_uint4(__float_as_uint(p.x), __float_as_uint(p.y), __float_as_uint(p.z),
                                         ebias[0] | (ebias[1] << 8) | (ebias[2] << 16) | (imask << 24));
        *reinterpret_cast<uint2*>(C.nodes + 5u * wnode + 1) = make_uint2(child_base, tri_base);
    }
    if (inner) {
        C.task_ref[qpos + rank] = ref;
        C.task_node[qpos + rank] = child_base + rank;
    } else if (used) {
        const uint32_t f = ref_first(T, ref);
        uint32_t src[4];      // a leaf has at most 4 triangles
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) src[k] = k < c ? T.perm[f + k] : 0u;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            if (k >= c) continue;
            const uint32_t dst = tri_base + toff + k;
            C.out_tris[3u * dst + 0] = C.in_tris[3u * src[k] + 0];
            C.out_tris[3u * dst + 1] = C.in_tris[3u * src[k] + 1];
            C.out_tris[3u * dst + 2] = C.in_tris[3u * src[k] + 2];
        }
    }
}

// one level of the wide tree: the tasks levels[l] .. levels[l + 1] - 1 of the queue (a ring of 8
// level starts); they append the next level's
__global__ void __launch_bounds__(128) k_collapse(CollapseCtx C, const uint32_t* levels, uint32_t l) {
    const uint32_t qbeg = levels[l & 7u], qend = levels[(l + 1u) & 7u];
    const uint32_t gl = threadIdx.x & 7u, gbase = threadIdx.x & 24u, gm = 0xffu << gbase;
    for (uint32_t ti = qbeg + ((blockIdx.x * blockDim.x + threadIdx.x) >> 3); ti < qend; ti += (gridDim.x * blockDim.x) >> 3)
        collapse_task(C, ti, gl, gm, gbase);
}
__global__ void k_collapse_next(const uint32_t* counters, uint32_t* levels, uint32_t l) {
    levels[(l + 2u) & 7u] = counters[2];
}

template <typename T>
static cudaError_t dalloc(T** p, size_t n) {
    return cudaMalloc((void**)p, std::max<size_t>(n, 1) * sizeof(T));
}

pt_status pt_build_bvh_impl(pt_scene* s, uint32_t leaf_size, uint32_t builder, uint32_t collapse, float tri_cost,
                            float box_cost, uint32_t max_width, cudaStream_t st) {
    const uint32_t n = s->n_tris;
    if (s->d_nodes) { cudaFree(s->d_nodes); s->d_nodes = nullptr; }
    if (s->d_tris) { cudaFree(s->d_tris); s->d_tris = nullptr; }
    // all scratch in one allocation (about 30 separate ones and their frees cost more than the
    // kernels of a small build)
    const uint32_t nblocks = (n + RS_TILE - 1) / RS_TILE;
    const bool ploc = builder == PT_BVH_PLOC;
    size_t used = 0;
    auto reserve = [&](size_t bytes) {
        const size_t at = used;
        used += (std::max<size_t>(bytes, 1) + 255) & ~(size_t)255;
        return at;
    };
    const size_t u32n = (size_t)n * sizeof(uint32_t), f4n = (size_t)n * sizeof(float4);
    const size_t o_k0 = reserve(2 * u32n), o_k1 = reserve(2 * u32n), o_v0 = reserve(u32n), o_v1 = reserve(u32n);
    const size_t o_hist = reserve((size_t)257 * nblocks * sizeof(uint32_t)), o_total = reserve(256 * sizeof(uint32_t));
    const size_t o_cb = reserve(8 * sizeof(uint32_t));
    const size_t o_left = reserve(u32n), o_right = reserve(u32n), o_pint = reserve(u32n), o_pleaf = reserve(u32n);
    const size_t o_first = reserve(u32n), o_last = reserve(u32n), o_flags = reserve(u32n);
    const size_t o_tref = reserve(u32n + 4), o_tnode = reserve(u32n + 4);
    const size_t o_counters = reserve(16 * sizeof(uint32_t)), o_state = reserve(8 * sizeof(PlocState));
    const size_t o_blo = reserve(f4n), o_bhi = reserve(f4n);
    const size_t o_clo = reserve(ploc ? 2 * f4n : 0), o_chi = reserve(ploc ? 2 * f4n : 0);
    const bool optimal = collapse == PT_COLLAPSE_OPTIMAL;
    const size_t o_dpc = reserve(optimal ? (size_t)8 * n * sizeof(float) : 0), o_dpd = reserve(optimal ? u32n : 0);
    unsigned char* scratch = nullptr;
    pt_status status = PT_OK;
    auto cleanup = [&]() {
        if (scratch) cudaFree(scratch);
    };
#define BTRY(call)                                                                           \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess) {                                                             \
            pt_set_error(std::string(#call) + ": " + cudaGetErrorString(e_));                \
            cleanup();                                                                       \
            return e_ == cudaErrorMemoryAllocation ? PT_ERR_OOM : PT_ERR_CUDA;               \
        }                                                                                    \
    } while (0)
    BTRY(dalloc(&scratch, used));
    auto u32 = [&](size_t o) { return reinterpret_cast<uint32_t*>(scratch + o); };
    auto f4 = [&](size_t o) { return reinterpret_cast<float4*>(scratch + o); };
    uint64_t *k0 = reinterpret_cast<uint64_t*>(scratch + o_k0), *k1 = reinterpret_cast<uint64_t*>(scratch + o_k1);
    uint32_t *v0 = u32(o_v0), *v1 = u32(o_v1), *hist = u32(o_hist), *total = u32(o_total), *cb = u32(o_cb);
    uint32_t *left = u32(o_left), *right = u32(o_right), *pint = u32(o_pint), *pleaf = u32(o_pleaf);
    uint32_t *first = u32(o_first), *last = u32(o_last), *flags = u32(o_flags);
    uint32_t *tref = u32(o_tref), *tnode = u32(o_tnode), *counters = u32(o_counters);
    uint32_t* levels = counters + 8;
    PlocState* state = reinterpret_cast<PlocState*>(scratch + o_state);
    float4 *blo = f4(o_blo), *bhi = f4(o_bhi), *clo = f4(o_clo), *chi = f4(o_chi);
    DpArrays D{nullptr, nullptr, leaf_size, tri_cost, box_cost, max_width};
    if (optimal) {
        D.cost = reinterpret_cast<float*>(scratch + o_dpc);
        D.dec = u32(o_dpd);
    }
    BTRY(dalloc(&s->d_nodes, (size_t)5 * (n + 1)));
    BTRY(dalloc(&s->d_tris, (size_t)3 * n));

    const uint32_t cbinit[6] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u};
    BTRY(cudaMemcpyAsync(cb, cbinit, sizeof(cbinit), cudaMemcpyHostToDevice, st));
    const uint32_t g = (n + 255) / 256;
    PT_LAUNCH(k_centroid_bounds, std::min<uint32_t>(g, (uint32_t)pt_num_sms() * 8u), 256, 0, st, s->d_tris_raw, n, cb);
    PT_LAUNCH(k_morton, g, 256, 0, st, s->d_tris_raw, n, cb, k0, v0);
    s->launches += 2;
    for (int pass = 0; pass < 8; ++pass) {
        const int shift = 8 * pass;
        PT_LAUNCH(k_rs_hist, nblocks, RS_THREADS, 0, st, k0, n, shift, hist, nblocks);
        PT_LAUNCH(k_rs_scan, 256, 256, 0, st, hist, nblocks, total);
        PT_LAUNCH(k_rs_scatter, nblocks, RS_THREADS, 0, st, k0, v0, k1, v1, n, shift, hist, total, nblocks);
        std::swap(k0, k1);
        std::swap(v0, v1);
        s->launches += 3;
    }
    BinTree T;
    T.left = left; T.right = right; T.first = first; T.last = last; T.perm = v0;
    T.blo = blo; T.bhi = bhi; T.tris = s->d_tris_raw;
    if (n > 1 && builder == PT_BVH_LBVH) {
        PT_LAUNCH(k_karras, (n - 1 + 255) / 256, 256, 0, st, k0, (int)n, left, right, pint, pleaf, first, last);
        BTRY(cudaMemsetAsync(flags, 0, (size_t)n * sizeof(uint32_t), st));
        PT_LAUNCH(k_bottom_up, g, 256, 0, st, T, (int)n, pint, pleaf, flags, D);
        s->launches += 2;
    } else if (n > 1) {
        // PLOC over the Morton order: cluster arrays ping-pong between (tref, flags, clo, chi)
        // and (tnode, last, clo + n, chi + n); scan prefixes in k1, block totals in hist,
        // nearest neighbours in pint, node triangle counts in pleaf, the final order in v1
        Clusters ca{tref, flags, clo, chi}, cb2{tnode, last, clo + n, chi + n};
        uint64_t* pre = k1;
        uint64_t* bsum = reinterpret_cast<uint64_t*>(hist);
        PT_LAUNCH(k_ploc_init, g, 256, 0, st, s->d_tris_raw, v0, n, ca);
        s->launches++;
        const PlocTree PT{left, right, pleaf, first, last, v1, blo, bhi};
        std::vector<PlocState> rounds;      // state before each round outside the tail
        PlocState now{n, 0u};
        BTRY(cudaMemcpyAsync(state, &now, sizeof(now), cudaMemcpyHostToDevice, st));
        uint32_t r = 0;
        while (now.m > PLOC_TAIL) {
            // grids for the clusters known to be left; later rounds of the batch have fewer
            const uint32_t m = now.m, nb = (m + PLOC_SCAN_TILE - 1) / PLOC_SCAN_TILE;
            Clusters x = ca, y = cb2;
            for (uint32_t k = 0; k < PLOC_BATCH; ++k) {
                const PlocState* cur = state + ((r + k) & 7u);
                PT_LAUNCH(k_ploc_nn, (m + PLOC_THREADS - 1) / PLOC_THREADS, PLOC_THREADS, 0, st, x, cur, pint);
                PT_LAUNCH(k_ploc_scan, nb, PLOC_THREADS, 0, st, pint, cur, pre, bsum);
                PT_LAUNCH(k_ploc_scan_top, 1, 1024, 0, st, bsum, cur, state + ((r + k + 1u) & 7u));
                PT_LAUNCH(k_ploc_compact, (m + 255) / 256, 256, 0, st, x, y, pint, cur, pre, bsum, n, left, right,
                          pleaf, blo, bhi, D);
                s->launches += 4;
                std::swap(x, y);
            }
            PlocState ring[8];
            BTRY(cudaMemcpyAsync(ring, state, sizeof(ring), cudaMemcpyDeviceToHost, st));
            BTRY(cudaStreamSynchronize(st));
            for (uint32_t k = 0; k < PLOC_BATCH && now.m > PLOC_TAIL; ++k) {
                const PlocState nx = ring[(r + k + 1u) & 7u];
                if (nx.m >= now.m || nx.m == 0u || nx.merged + nx.m != n) {
                    pt_set_error("PLOC clustering made no progress");
                    cleanup();
                    return PT_ERR_CUDA;
                }
                rounds.push_back(now);
                now = nx;
                std::swap(ca, cb2);
            }
            r += PLOC_BATCH;
        }
        static_assert(PLOC_TAIL <= 2 * PLOC_TAIL_THREADS && PLOC_BATCH <= 4, "two clusters a thread; the ring holds a batch");
        BTRY(cudaFuncSetAttribute(k_ploc_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PLOC_TAIL_SMEM));
        PT_LAUNCH(k_ploc_tail, 1, PLOC_TAIL_THREADS, PLOC_TAIL_SMEM, st, ca, now.m, now.merged, n, PT, D, counters);
        s->launches++;
        uint32_t done = 0;
        BTRY(cudaMemcpyAsync(&done, counters, sizeof(done), cudaMemcpyDeviceToHost, st));
        BTRY(cudaStreamSynchronize(st));
        if (!done) {
            pt_set_error("PLOC clustering made no progress");
            cleanup();
            return PT_ERR_CUDA;
        }
        for (size_t q = rounds.size(); q-- > 0;) {
            const uint32_t merged_after = q + 1 < rounds.size() ? rounds[q + 1].merged : now.merged;
            const uint32_t lo = n - 1u - merged_after, hi = n - 2u - rounds[q].merged;
            PT_LAUNCH(k_ploc_layout, (hi - lo + 1 + 255) / 256, 256, 0, st, lo, hi, PT);
            s->launches++;
        }
        T.perm = v1;
    }
    // collapse, one level per launch
    const uint32_t root_ref = n > 1 ? 0u : LEAF_BIT;
    const uint32_t init[4] = {1u, 0u, 1u, 0u};
    BTRY(cudaMemcpyAsync(counters, init, sizeof(init), cudaMemcpyHostToDevice, st));
    const uint32_t zero = 0;
    BTRY(cudaMemcpyAsync(tref, &root_ref, sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    BTRY(cudaMemcpyAsync(tnode, &zero, sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    CollapseCtx C;
    C.T = T;
    C.leaf_size = leaf_size;
    C.width = max_width;
    C.task_ref = tref;
    C.task_node = tnode;
    C.counters = counters;
    C.nodes = s->d_nodes;
    C.out_tris = s->d_tris;
    C.in_tris = s->d_tris_raw;
    C.dp = D;
    // the levels run without the host, four between read-backs of the queue: a level has at most
    // max_width times the tasks of the one before it
    const uint32_t level_init[8] = {0u, 1u, 0u, 0u, 0u, 0u, 0u, 0u};
    BTRY(cudaMemcpyAsync(levels, level_init, sizeof(level_init), cudaMemcpyHostToDevice, st));
    uint32_t depth = 0, l = 0;
    uint64_t width_ub = 1;
    uint32_t host_counters[16] = {0};
    for (bool more = true; more;) {
        for (uint32_t k = 0; k < 4; ++k, ++l) {
            const uint32_t grid = (uint32_t)std::min<uint64_t>((width_ub + 15) / 16, (uint64_t)pt_num_sms() * 16);
            PT_LAUNCH(k_collapse, grid, 128, 0, st, C, levels, l);
            PT_LAUNCH(k_collapse_next, 1, 1, 0, st, counters, levels, l);
            s->launches += 2;
            width_ub = std::min<uint64_t>(width_ub * max_width, n);
        }
        BTRY(cudaMemcpyAsync(host_counters, counters, sizeof(host_counters), cudaMemcpyDeviceToHost, st));
        BTRY(cudaStreamSynchronize(st));
        for (uint32_t k = l - 4; k < l && more; ++k) {
            if (host_counters[8 + (k & 7u)] < host_counters[8 + ((k + 1u) & 7u)]) ++depth;
            else more = false;
        }
        if (depth > 200) { pt_set_error("BVH collapse did not terminate"); status = PT_ERR_CUDA; break; }
    }
    BTRY(cudaGetLastError());
    if (status == PT_OK && host_counters[1] != n) {
        pt_set_error("BVH collapse placed " + std::to_string(host_counters[1]) + " of " + std::to_string(n) + " triangles");
        status = PT_ERR_CUDA;
    }
    s->n_nodes = host_counters[0];
    s->depth = depth;
    cleanup();
#undef BTRY
    return status;
}

// ------------------------------------------------------------------ environment tables
// weights w = luminance * sin(theta at the texel centre); per-row conditional CDF and the
// marginal CDF over rows; a row (or the whole map) of zero weight gets a uniform CDF.
__global__ void k_env_rows(const float* env, int w, int h, float* wtex, float* cond, float* rowsum) {
    __shared__ float part[256];
    __shared__ float running;
    const int y = blockIdx.x;
    const float st = sinf(PT_PI_F * ((float)y + 0.5f) / (float)h);
    if (threadIdx.x == 0) running = 0.0f;
    __syncthreads();
    float* cd = cond + (size_t)y * (w + 1);
    for (int base = 0; base < w; base += 256) {
        const int x = base + threadIdx.x;
        float wt = 0.0f;
        if (x < w) {
            const float* t = env + 3 * ((size_t)y * w + x);
            wt = fmaxf(lum3(mk3(t[0], t[1], t[2])) * st, 0.0f);
            wtex[(size_t)y * w + x] = wt;
        }
        part[threadIdx.x] = wt;
        __syncthreads();
        for (int off = 1; off < 256; off <<= 1) {
            const float v = threadIdx.x >= (unsigned)off ? part[threadIdx.x - off] : 0.0f;
            __syncthreads();
            part[threadIdx.x] += v;
            __syncthreads();
        }
        if (x < w) cd[x + 1] = running + part[threadIdx.x];
        __syncthreads();
        if (threadIdx.x == 0) running += part[255];
        __syncthreads();
    }
    const float tot = running;
    for (int x = threadIdx.x; x < w; x += 256) cd[x + 1] = tot > 0.0f ? cd[x + 1] / tot : (float)(x + 1) / (float)w;
    if (threadIdx.x == 0) {
        cd[0] = 0.0f;
        rowsum[y] = tot;
    }
}

__global__ void k_env_marg(const float* rowsum, int h, float* marg, float* total) {
    __shared__ float part[1024];
    __shared__ float running;
    if (threadIdx.x == 0) running = 0.0f;
    __syncthreads();
    for (int base = 0; base < h; base += 1024) {
        const int y = base + threadIdx.x;
        part[threadIdx.x] = y < h ? rowsum[y] : 0.0f;
        __syncthreads();
        for (int off = 1; off < 1024; off <<= 1) {
            const float v = threadIdx.x >= (unsigned)off ? part[threadIdx.x - off] : 0.0f;
            __syncthreads();
            part[threadIdx.x] += v;
            __syncthreads();
        }
        if (y < h) marg[y + 1] = running + part[threadIdx.x];
        __syncthreads();
        if (threadIdx.x == 0) running += part[1023];
        __syncthreads();
    }
    const float tot = running;
    for (int y = threadIdx.x; y < h; y += 1024) marg[y + 1] = tot > 0.0f ? marg[y + 1] / tot : (float)(y + 1) / (float)h;
    if (threadIdx.x == 0) {
        marg[0] = 0.0f;
        total[0] = tot;
    }
}

// search guides: guide[g] = the CDF index for u = g / G (see cdf_find_guided)
__global__ void k_env_guides(const float* marg, const float* cond, int w, int h, int gm, int gc, int* guide) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t <= gm) {
        guide[t] = cdf_find(marg, h, (float)t / (float)gm);
        return;
    }
    const int r = t - (gm + 1);
    if (r >= h * (gc + 1)) return;
    const int y = r / (gc + 1), g = r % (gc + 1);
    guide[t] = cdf_find(cond + (size_t)y * (w + 1), w, (float)g / (float)gc);
}

pt_status pt_build_env_impl(pt_scene* s, cudaStream_t st) {
    if (!s->d_env || s->env_w <= 0) { s->env_total = 0.0f; return PT_OK; }
    const int w = s->env_w, h = s->env_h;
    float* rowsum = nullptr;
    if (!s->d_env_wtex) {
        PT_CUDA_TRY(cudaMalloc(&s->d_env_wtex, (size_t)w * h * sizeof(float)));
        PT_CUDA_TRY(cudaMalloc(&s->d_env_cond, (size_t)h * (w + 1) * sizeof(float)));
        PT_CUDA_TRY(cudaMalloc(&s->d_env_marg, (size_t)(h + 1) * sizeof(float)));
        PT_CUDA_TRY(cudaMalloc(&s->d_env_total, sizeof(float)));
        int gm = 1, gc = 1;
        while (gm < h) gm <<= 1;
        while (gc < w) gc <<= 1;
        s->env_gm = gm;
        s->env_gc = gc;
        PT_CUDA_TRY(cudaMalloc(&s->d_env_guide, ((size_t)gm + 1 + (size_t)h * (gc + 1)) * sizeof(int)));
    }
    PT_CUDA_TRY(cudaMalloc(&rowsum, (size_t)h * sizeof(float)));
    PT_LAUNCH(k_env_rows, h, 256, 0, st, s->d_env, w, h, s->d_env_wtex, s->d_env_cond, rowsum);
    PT_LAUNCH(k_env_marg, 1, 1024, 0, st, rowsum, h, s->d_env_marg, s->d_env_total);
    const int ng = s->env_gm + 1 + h * (s->env_gc + 1);
    PT_LAUNCH(k_env_guides, (ng + 255) / 256, 256, 0, st, s->d_env_marg, s->d_env_cond, w, h, s->env_gm, s->env_gc,
              s->d_env_guide);
    s->launches += 3;
    PT_CUDA_TRY(cudaMemcpyAsync(&s->env_total, s->d_env_total, sizeof(float), cudaMemcpyDeviceToHost, st));
    PT_CUDA_TRY(cudaStreamSynchronize(st));
    cudaFree(rowsum);
    return PT_OK;
}
