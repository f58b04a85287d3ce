// Gather into key order and the linear octree over the key-ordered particles
// (Sec. 1.2: an octree divides the volume; particles follow the Hilbert curve, so
// every octree cell is one contiguous range of the sorted order).
#include <algorithm>

#include "sph_internal.cuh"

namespace sphgrp {

// x * 2^32 is exact; its floor is the fixed-point coordinate, the remainder (exact in
// FP64, < 1) keeps the rest of the position and is rounded once to FP32.  For
// 2^-32 <= x < 1 both come from the bits of x with integer operations (FP64 arithmetic
// is a slow pipe on this part): x 2^32 = M 2^-s with M = 2^52 + f and s = 1043 - e in
// [21, 52], so the floor is M >> s and the remainder (M mod 2^s) 2^-s, whose integer
// part converts to FP32 with one rounding and scales by 2^-s exactly.  Other x take
// the FP64 form.
__device__ __forceinline__ uint32_t fix_split(double x, float& rem) {
    const uint64_t b = __double_as_longlong(x);
    const int e = (int)(b >> 52);   // biased exponent; the sign bit makes it >= 2048
    const int s = 1043 - e;
    if (s >= 21 && s <= 52) {
        const uint64_t M = (b & 0xfffffffffffffull) | (1ull << 52);
        rem = __ull2float_rn(M & ((1ull << s) - 1ull)) * __int_as_float((127 - s) << 23);
        return (uint32_t)(M >> s);
    }
    const double sx = x * kBoxToUnit, fx = floor(sx);
    rem = (float)(sx - fx);
    return (uint32_t)fx;
}

// pos/m (original order) -> key-ordered FP64 copies and the fixed-point layout.
__global__ void k_gather(int64_t n, const int32_t* __restrict__ perm, const double* __restrict__ pos,
                         const float* __restrict__ m, double* __restrict__ xd, double* __restrict__ yd,
                         double* __restrict__ zd, uint4* __restrict__ pfix, float4* __restrict__ poff) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    int i = perm[r];
    double x = pos[3 * (int64_t)i], y = pos[3 * (int64_t)i + 1], z = pos[3 * (int64_t)i + 2];
    float ox, oy, oz;
    uint4 P;
    P.x = fix_split(x, ox);
    P.y = fix_split(y, oy);
    P.z = fix_split(z, oz);
    P.w = 0u;
    pfix[r] = P;
    poff[r] = make_float4(ox, oy, oz, m[i]);
    xd[r] = x;
    yd[r] = y;
    zd[r] = z;
}

// The octree of one or many boxes (a forest) straight from the sorted keys, without a pass per
// level.  A node is a cell whose parent holds more than `leaf` particles, named by its
// first particle i and its level l.  A cell of level l starts at i iff the keys of i and
// i - 1 share fewer than l digits; call the first such level dl(i) (0 at the start of a
// box).  A cell holds more than `leaf` particles iff leaf + 1 consecutive ones lie in it, so
// the deepest level at which the cell of i does is
//   c(i) = max over w in [i - leaf, i] of the digits shared by the keys of w and w + leaf,
// and the nodes starting at i are those of the levels dl(i) .. e(i) = min(c(i) + 1, 21).
// Their ids are ordered by (level, first particle): counted per level and tile of particles,
// one scan, written by a second pass.  So a level's nodes are contiguous, a node's children
// are contiguous, and its first child starts where it starts.
//
// Bound by the particles' keys (read twice) on large sets, by its five launches on small
// ones.  A kernel per level, every node searching its octants' bounds, spent 5-30 us on
// each of a dozen levels (keys, order and octree of 4.0M particles 1.10 -> 1.02 ms, differentiable forces of 30k 1.94 -> 1.85 ms).

constexpr int kTreeTile = 256;        // particles per tile (a warp's in k_tree_nodes)
constexpr int kTreeBlock = 4;         // tiles per block of k_tree_marks
constexpr int kMaxLeaf = 1024;        // largest leaf size

struct TreeArgs {
    const uint64_t* keys;
    int64_t n;
    int nbox;
    const int64_t* box_off;       // null: one box
    const int32_t* box_of_rank;   // null: one box
    const int32_t* box_cfg;       // bits 16..23: the box's leaf size (0: leaf_size); null: leaf_size
    int leaf_size;
    int halo;                     // largest leaf size of any box
    int64_t cap;
    int32_t* marks;               // per particle: dl | e << 8
    int32_t* first_id;            // per particle: id of the shallowest node that starts there
    int32_t* blk;                 // nodes per (level, tile), then their exclusive scan and the total
    int64_t ntile;
    int32_t* lcnt;
    int4* nlink;
    float4* next;
    int32_t* nlevel;
    int32_t* nparent;
    uint32_t* narrive;
    unsigned* err;
};

// digits (3 bits, from the top of 63) shared by two keys
__device__ __forceinline__ int shared_digits(uint64_t a, uint64_t b) {
    const uint64_t x = a ^ b;
    return x == 0 ? kKeyLevels : (__clzll((long long)x) - 1) / 3;
}

struct BoxRange {
    int64_t lo, hi;
    int leaf;
};

__device__ __forceinline__ BoxRange box_range(const TreeArgs& a, int64_t i) {
    if (!a.box_off) return BoxRange{0, a.n, a.leaf_size};
    const int b = a.box_of_rank[i];
    int leaf = a.leaf_size;
    if (a.box_cfg) {
        const int lb = (a.box_cfg[b] >> 16) & 0xff;
        if (lb > 0) leaf = lb;
    }
    return BoxRange{a.box_off[b], a.box_off[b + 1], leaf};
}

// dl and e of every particle, and each tile's nodes per level
__global__ void __launch_bounds__(kTreeTile) k_tree_marks(TreeArgs a) {
    constexpr int kPart = kTreeBlock * kTreeTile;
    __shared__ int8_t s1[kPart + kMaxLeaf + 16];   // digits shared by the keys of w and w + leaf (-1: not one box)
    __shared__ int8_t s8[kPart + kMaxLeaf + 16];   // the largest of eight in a row
    __shared__ int cnt[kTreeBlock][kTreeLevels];
    const int64_t part0 = blockIdx.x * (int64_t)kPart;
    const int len = kPart + a.halo;                // entry k stands for w = part0 - halo + k
    for (int k = threadIdx.x; k < kTreeBlock * kTreeLevels; k += kTreeTile) (&cnt[0][0])[k] = 0;
    for (int k = threadIdx.x; k < len + 8; k += kTreeTile) {
        const int64_t w = part0 - a.halo + k;
        int v = -1;
        if (k < len && w >= 0 && w < a.n) {
            const BoxRange B = box_range(a, w);
            if (w + B.leaf < B.hi) v = shared_digits(a.keys[w], a.keys[w + B.leaf]);
        }
        s1[k] = (int8_t)v;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < len; k += kTreeTile) {
        int v = s1[k];
#pragma unroll
        for (int q = 1; q < 8; ++q) v = max(v, (int)s1[k + q]);
        s8[k] = (int8_t)v;
    }
    __syncthreads();
    for (int t = 0; t < kTreeBlock; ++t) {
        const int64_t i = part0 + t * kTreeTile + threadIdx.x;
        if (i >= a.n) break;
        const BoxRange B = box_range(a, i);
        const int dl = i == B.lo ? 0 : 1 + shared_digits(a.keys[i - 1], a.keys[i]);
        const int w1 = a.halo + t * kTreeTile + threadIdx.x;
        int w = w1 - (int)min((int64_t)B.leaf, i - B.lo);
        int c = -1;
        for (; w + 7 <= w1; w += 8) c = max(c, (int)s8[w]);
        for (; w <= w1; ++w) c = max(c, (int)s1[w]);
        const int e = min(c + 1, kKeyLevels);
        a.marks[i] = dl | e << 8;
        for (int l = dl; l <= e; ++l) atomicAdd(&cnt[t][l], 1);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kTreeBlock * kTreeLevels; k += kTreeTile) {
        const int t = k / kTreeLevels, l = k - t * kTreeLevels;
        const int64_t tile = blockIdx.x * (int64_t)kTreeBlock + t;
        if (tile < a.ntile) a.blk[l * a.ntile + tile] = cnt[t][l];
    }
}

// first id of level l (l = kTreeLevels: the number of nodes)
__device__ __forceinline__ int level_first(const TreeArgs& a, int l) { return a.blk[l * a.ntile]; }

// Ids of every particle's nodes, linked down to their first child: a warp per tile, lane l
// holding the next id of level l.  With more nodes than the arrays hold, only the roots are
// made, as leaves, and the error flag is set (the caller builds again, or makes no search
// and reports it); lcnt[kTreeLevels] tells how many there would be.
__global__ void __launch_bounds__(256) k_tree_nodes(TreeArgs a) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const int total = level_first(a, kTreeLevels);
    const bool fits = total <= a.cap;
    if (blockIdx.x == 0 && threadIdx.x <= kTreeLevels) {
        const int l = threadIdx.x;
        if (l == kTreeLevels) a.lcnt[l] = total;
        else if (fits) a.lcnt[l] = level_first(a, l + 1) - level_first(a, l);
        else a.lcnt[l] = l == 0 ? a.nbox : 0;
        if (!fits && l == 0) atomicOr(a.err, kErrNodes);
    }
    const int64_t tile = (blockIdx.x * 256ll + threadIdx.x) >> 5;
    if (tile >= a.ntile) return;
    int run = lane < kTreeLevels ? a.blk[lane * a.ntile + tile] : 0;
    for (int r = 0; r < kTreeTile / 32; ++r) {
        const int64_t i = tile * kTreeTile + r * 32 + lane;
        int dl = kTreeLevels, e = -1;
        if (i < a.n) {
            const int m = a.marks[i];
            dl = m & 0xff;
            e = m >> 8;
        }
        const bool starts = dl <= e;
        const int l0 = __reduce_min_sync(0xffffffffu, starts ? dl : kTreeLevels);
        const int l1 = __reduce_max_sync(0xffffffffu, starts ? e : -1);
        int up = -1;   // the node of the level above that starts here
        for (int l = l0; l <= l1; ++l) {
            const bool have = dl <= l && l <= e;
            const unsigned b = __ballot_sync(0xffffffffu, have);
            const int first = __shfl_sync(0xffffffffu, run, l);
            if (lane == l) run += __popc(b);
            if (!have) continue;
            const int id = first + __popc(b & lt);
            if (l == dl) a.first_id[i] = id;
            if (fits || l == 0) {
                a.nlink[id] = make_int4((int)i, 0, -1, -1);
                a.nlevel[id] = l;
                a.narrive[id] = 0u;
                if (up >= 0) a.nlink[up].z = id;
            }
            up = id;
        }
    }
}

// A node's particle count, its children's number and parent, and its skip pointer.  Its range
// ends where its next sibling starts; a last sibling's end is searched in the keys.
__global__ void __launch_bounds__(256) k_tree_link(TreeArgs a) {
    const int total = level_first(a, kTreeLevels);
    const bool fits = total <= a.cap;
    const int nn = fits ? total : a.nbox;
    int* link = reinterpret_cast<int*>(a.nlink);   // .y and .w are written, .x and .z only read
    for (int id = blockIdx.x * 256 + threadIdx.x; id < nn; id += gridDim.x * 256) {
        const int64_t i = link[4ll * id];
        const int l = a.nlevel[id];
        const BoxRange B = box_range(a, i);
        int64_t end = B.hi;
        if (l > 0) {
            const uint64_t k = a.keys[i];
            int64_t j = -1;
            if (id + 1 < level_first(a, l + 1)) {
                const int64_t s = link[4ll * (id + 1)];
                if (s < B.hi && shared_digits(k, a.keys[s]) >= l - 1) j = s;
            }
            if (j < 0) {
                // first particle outside the cell: doubling steps, then halving
                int64_t in = i, step = 1;
                while (in + step < B.hi && shared_digits(k, a.keys[in + step]) >= l) {
                    in += step;
                    step *= 2;
                }
                int64_t out = min(in + step, B.hi);
                while (out - in > 1) {
                    const int64_t mid = (in + out) >> 1;
                    if (shared_digits(k, a.keys[mid]) >= l) in = mid; else out = mid;
                }
                j = out;
            }
            end = j;
        } else {
            a.nparent[id] = -1;
        }
        const int c0 = fits ? link[4ll * id + 2] : -1;
        int nc = 0;
        if (c0 >= 0) {
            const int last = level_first(a, l + 2);   // one past the children's level
            for (nc = 1; nc < 8 && c0 + nc < last && link[4ll * (c0 + nc)] < end; ++nc) {}
            for (int c = 0; c < nc; ++c) a.nparent[c0 + c] = id;
        }
        a.next[id] = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(nc));
        link[4ll * id + 1] = (int)(end - i);
        link[4ll * id + 3] = fits && end < B.hi ? a.first_id[end] : -1;
    }
}

// first node and number of nodes of a level
__device__ __forceinline__ void level_range(const int32_t* __restrict__ lcnt, int level, int64_t cap, int& a, int& nf) {
    int64_t first = 0;
    for (int l = 0; l < level; ++l) first += lcnt[l];
    a = (int)min(first, cap);
    nf = (int)max((int64_t)0, min((int64_t)lcnt[level], cap - first));
}

// Box -> centre (fixed point) and padded half extents.  Particles of the node lie in
// [lo, hi + 1) units; with the centre rounded down to a whole unit the half extent
// (hi - lo + 2) / 2 covers that interval.  Extents are rounded up.
__device__ __forceinline__ void write_box(int id, uint4 l, uint4 h, float hmax, uint4* __restrict__ blo,
                                          uint4* __restrict__ bhi, uint4* __restrict__ ncen,
                                          float4* __restrict__ next) {
    blo[id] = l;
    bhi[id] = h;
    const uint64_t wx = (uint64_t)h.x - l.x + 1, wy = (uint64_t)h.y - l.y + 1, wz = (uint64_t)h.z - l.z + 1;
    ncen[id] = make_uint4(l.x + (uint32_t)(wx >> 1), l.y + (uint32_t)(wy >> 1), l.z + (uint32_t)(wz >> 1),
                          __float_as_uint(hmax));
    float* e = reinterpret_cast<float*>(next + id);   // .w (the child count) is read meanwhile
    e[0] = __fmul_ru(__ull2float_ru(wx + 1), 0.5f);
    e[1] = __fmul_ru(__ull2float_ru(wy + 1), 0.5f);
    e[2] = __fmul_ru(__ull2float_ru(wz + 1), 0.5f);
}

// What a node takes from its particles (a leaf) or its children: tight box (BOXES) and hmax.
struct NodeBox {
    uint4 l, h;
    float hm;
};

// children [c0, c0 + nc), read past the L1 cache (they may have been written by this launch)
template <bool BOXES>
__device__ __forceinline__ NodeBox box_of_children(int c0, int nc, const uint4* blo, const uint4* bhi,
                                                   const uint4* ncen) {
    NodeBox b{make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0u), make_uint4(0u, 0u, 0u, 0u), 0.0f};
    for (int c = c0; c < c0 + nc; ++c) {
        if (BOXES) {
            const uint4 cl = __ldcg(blo + c), ch = __ldcg(bhi + c);
            b.l.x = min(b.l.x, cl.x); b.l.y = min(b.l.y, cl.y); b.l.z = min(b.l.z, cl.z);
            b.h.x = max(b.h.x, ch.x); b.h.y = max(b.h.y, ch.y); b.h.z = max(b.h.z, ch.z);
        }
        b.hm = fmaxf(b.hm, __ldcg(reinterpret_cast<const float*>(ncen + c) + 3));
    }
    return b;
}

template <bool BOXES>
__device__ __forceinline__ void write_node(int id, const NodeBox& b, uint4* blo, uint4* bhi, uint4* ncen,
                                           float4* next) {
    if (BOXES) write_box(id, b.l, b.h, b.hm, blo, bhi, ncen, next);
    else reinterpret_cast<float*>(ncen + id)[3] = b.hm;
}

// The leaves, eight lanes to one.  CLIMB: the first lane then goes up, the last child to
// arrive at a node completing it and going on; the arrival counters wrap to zero by
// themselves.  Maxima and minima do not depend on the order.
//
// Climbing takes one launch where a launch per level spends 6-10 us on each level of a few
// nodes (hmax of a 131k tree 81 -> 32 us, boxes of a 30k one 100 -> 40 us), but its fences
// make it slow on many nodes (16.8M particles: boxes 1.35 ms, hmax 0.70 ms): trees above
// kClimbNodes nodes take a launch per level above the leaves (k_tree_level).
template <bool BOXES, bool CLIMB>
__global__ void __launch_bounds__(256) k_tree_leaves(const int32_t* __restrict__ lcnt, int64_t cap,
                                                     const int4* __restrict__ nlink, float4* next,
                                                     const uint4* __restrict__ pfix,
                                                     const int32_t* __restrict__ nparent, uint32_t* narrive,
                                                     uint4* blo, uint4* bhi, uint4* ncen) {
    int a, nf;
    level_range(lcnt, kTreeLevels - 1, cap, a, nf);
    const int nn = a + nf;
    const int sub = threadIdx.x & 7;
    for (int64_t base = (blockIdx.x * 256ll + threadIdx.x) >> 5 << 2; base < nn; base += gridDim.x * 32ll) {   // warp-uniform
        int id = (int)base + ((threadIdx.x & 31) >> 3);
        int4 L = make_int4(0, 0, 0, -1);
        if (id < nn) L = nlink[id];
        const bool leaf = id < nn && L.z < 0;
        NodeBox b{make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0u), make_uint4(0u, 0u, 0u, 0u), 0.0f};
        if (leaf) {
            for (int q = L.x + sub; q < L.x + L.y; q += 8) {
                if (BOXES) {
                    const uint4 P = pfix[q];
                    b.l.x = min(b.l.x, P.x); b.l.y = min(b.l.y, P.y); b.l.z = min(b.l.z, P.z);
                    b.h.x = max(b.h.x, P.x); b.h.y = max(b.h.y, P.y); b.h.z = max(b.h.z, P.z);
                    b.hm = fmaxf(b.hm, __uint_as_float(P.w));
                } else {
                    b.hm = fmaxf(b.hm, __uint_as_float(pfix[q].w));
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            if (BOXES) {
                b.l.x = min(b.l.x, __shfl_xor_sync(0xffffffffu, b.l.x, o));
                b.l.y = min(b.l.y, __shfl_xor_sync(0xffffffffu, b.l.y, o));
                b.l.z = min(b.l.z, __shfl_xor_sync(0xffffffffu, b.l.z, o));
                b.h.x = max(b.h.x, __shfl_xor_sync(0xffffffffu, b.h.x, o));
                b.h.y = max(b.h.y, __shfl_xor_sync(0xffffffffu, b.h.y, o));
                b.h.z = max(b.h.z, __shfl_xor_sync(0xffffffffu, b.h.z, o));
            }
            b.hm = fmaxf(b.hm, __shfl_xor_sync(0xffffffffu, b.hm, o));
        }
        if (leaf && sub == 0) {
            if (BOXES && L.y == 0) b.l = b.h = make_uint4(0u, 0u, 0u, 0u);
            write_node<BOXES>(id, b, blo, bhi, ncen, next);
            while (CLIMB) {
                const int p = nparent[id];
                if (p < 0) break;
                const int nc = __float_as_int(reinterpret_cast<const float*>(next + p)[3]);
                __threadfence();
                if (atomicInc(&narrive[p], (unsigned)nc - 1u) != (unsigned)nc - 1u) break;
                __threadfence();
                id = p;
                b = box_of_children<BOXES>(nlink[p].z, nc, blo, bhi, ncen);
                write_node<BOXES>(id, b, blo, bhi, ncen, next);
            }
        }
        __syncwarp();
    }
}

// the internal nodes of one level, from their children
template <bool BOXES>
__global__ void __launch_bounds__(256) k_tree_level(const int32_t* __restrict__ lcnt, int level, int64_t cap,
                                                    const int4* __restrict__ nlink, float4* next, uint4* blo,
                                                    uint4* bhi, uint4* ncen) {
    int a, nf;
    level_range(lcnt, level, cap, a, nf);
    for (int k = blockIdx.x * 256 + threadIdx.x; k < nf; k += gridDim.x * 256) {
        const int id = a + k;
        const int c0 = nlink[id].z;
        if (c0 < 0) continue;
        const int nc = __float_as_int(reinterpret_cast<const float*>(next + id)[3]);
        write_node<BOXES>(id, box_of_children<BOXES>(c0, nc, blo, bhi, ncen), blo, bhi, ncen, next);
    }
}

// Walk start tables (see kStartLevels), one per box: every node of levels 1 .. kStartLevels
// enters its box's table under its cell, found from any of its particles (the cell of
// level l is the top l bits of the fixed-point coordinates).  box_of_rank null: one box.
__global__ void k_start_table(const int32_t* __restrict__ lcnt, int64_t cap, const int4* __restrict__ nlink,
                              const int32_t* __restrict__ nlevel, const uint4* __restrict__ pfix,
                              const int32_t* __restrict__ box_of_rank, int32_t* __restrict__ tab) {
    int end, nf;
    level_range(lcnt, kStartLevels, cap, end, nf);
    end += nf;
    for (int id = lcnt[0] + blockIdx.x * blockDim.x + threadIdx.x; id < end; id += gridDim.x * blockDim.x) {
        const int l = nlevel[id];
        const int4 L = nlink[id];
        if (l < 1 || l > kStartLevels || L.y <= 0) continue;
        const uint4 P = pfix[L.x];
        const uint32_t x = P.x >> (32 - l), y = P.y >> (32 - l), z = P.z >> (32 - l);
        uint32_t m = 0;
        for (int b = l - 1; b >= 0; --b) m = (m << 3) | (((x >> b) & 1u) << 2) | (((y >> b) & 1u) << 1) | ((z >> b) & 1u);
        tab[(size_t)(box_of_rank ? box_of_rank[L.x] : 0) * kStartTableSize + start_table_offset(l) + m] = id;
    }
}

constexpr int kTreeGrid = 1024;   // most blocks of the grid-stride kernels

// Node arrays for cap nodes and the per-level counts, one block from the stream's memory pool
// (the old contents are dropped).  Ten arrays by cudaMalloc made a context's first build of
// 4.0M particles 1.37 ms where the second takes 0.41 (1.0M: 1.06 and 0.20); every cudaFree of
// an outgrown one would wait for the whole device.
int alloc_tree(Ctx* c, int64_t cap, cudaStream_t s) {
    Tree& t = c->tree;
    if (cap <= t.cap) return SPHGRP_OK;
    if (t.block) cudaFreeAsync(t.block, s);
    t.block = nullptr;
    t.cap = 0;
    const int64_t tiles = (c->n_max + kTreeTile - 1) / kTreeTile;
    const size_t counts = (kTreeLevels + 1) + (kTreeLevels * tiles + 1);
    const size_t bytes = (size_t)cap * (5 * sizeof(uint4) + 3 * sizeof(int32_t)) + counts * sizeof(int32_t);
    if (cudaMallocAsync(&t.block, bytes, s) != cudaSuccess) {
        t.block = nullptr;
        cudaGetLastError();
        return set_error(SPHGRP_ENOMEM, "octree allocation failed");
    }
    // the 16-byte records first, then the words
    t.ncen = static_cast<uint4*>(t.block);
    t.next = reinterpret_cast<float4*>(t.ncen + cap);
    t.nlink = reinterpret_cast<int4*>(t.next + cap);
    t.box_lo = reinterpret_cast<uint4*>(t.nlink + cap);
    t.box_hi = t.box_lo + cap;
    t.nlevel = reinterpret_cast<int32_t*>(t.box_hi + cap);
    t.nparent = t.nlevel + cap;
    t.narrive = reinterpret_cast<uint32_t*>(t.nparent + cap);
    t.level_cnt = reinterpret_cast<int32_t*>(t.narrive + cap);
    t.tile_cnt = t.level_cnt + kTreeLevels + 1;
    t.cap = cap;
    return SPHGRP_OK;
}

// Nodes of the octrees of nbox boxes (box_off null: one) in four launches and a scan; counts
// per level and in all on the device.
static int launch_nodes(Ctx* c, int nbox, const int64_t* box_off, const int32_t* box_of_rank, const int32_t* box_cfg,
                        cudaStream_t s) {
    Tree& t = c->tree;
    TreeArgs a;
    a.keys = c->keys;
    a.n = c->n;
    a.nbox = nbox;
    a.box_off = box_off;
    a.box_of_rank = box_of_rank;
    a.box_cfg = box_cfg;
    a.leaf_size = c->p.leaf_size;
    a.halo = box_cfg ? std::max(c->p.leaf_size, 255) : c->p.leaf_size;
    a.cap = t.cap;
    a.marks = c->flag;
    a.first_id = c->scan;
    a.blk = t.tile_cnt;
    a.ntile = (c->n + kTreeTile - 1) / kTreeTile;
    a.lcnt = t.level_cnt;
    a.nlink = t.nlink;
    a.next = t.next;
    a.nlevel = t.nlevel;
    a.nparent = t.nparent;
    a.narrive = t.narrive;
    a.err = c->err;
    k_tree_marks<<<(unsigned)((a.ntile + kTreeBlock - 1) / kTreeBlock), kTreeTile, 0, s>>>(a);
    note_launch();
    const int64_t words = kTreeLevels * a.ntile;
    int rc = exclusive_scan_i32(c, t.tile_cnt, t.tile_cnt, words, t.tile_cnt + words, s);
    if (rc) return rc;
    k_tree_nodes<<<(unsigned)((a.ntile + 7) / 8), 256, 0, s>>>(a);
    note_launch();
    const int64_t bound = std::min<int64_t>(t.cap, (int64_t)kTreeLevels * c->n);
    k_tree_link<<<(unsigned)std::min<int64_t>((bound + 255) / 256, 8 * kTreeGrid), 256, 0, s>>>(a);
    note_launch();
    return check_cuda(cudaGetLastError(), "octree nodes");
}

constexpr int64_t kClimbNodes = 1 << 17;

// Boxes and hmax (BOXES) or hmax alone, of at most `bound` nodes in levels 0 .. deepest.
template <bool BOXES>
static void launch_up(Ctx* c, int64_t bound, int deepest, cudaStream_t s) {
    Tree& t = c->tree;
    const int grid = (int)std::min<int64_t>((bound + 31) / 32, 16 * kTreeGrid);
    if (bound <= kClimbNodes) {
        k_tree_leaves<BOXES, true><<<grid, 256, 0, s>>>(t.level_cnt, t.cap, t.nlink, t.next, c->pfix, t.nparent,
                                                        t.narrive, t.box_lo, t.box_hi, t.ncen);
        note_launch();
        return;
    }
    k_tree_leaves<BOXES, false><<<grid, 256, 0, s>>>(t.level_cnt, t.cap, t.nlink, t.next, c->pfix, t.nparent,
                                                     t.narrive, t.box_lo, t.box_hi, t.ncen);
    note_launch();
    for (int level = deepest - 1; level >= 0; --level) {
        const int64_t most = level < 6 ? std::min<int64_t>(bound, (int64_t)t.nroots << (3 * level)) : bound;
        k_tree_level<BOXES><<<(int)std::min<int64_t>((most + 255) / 256, 2 * kTreeGrid), 256, 0, s>>>(
            t.level_cnt, level, t.cap, t.nlink, t.next, t.box_lo, t.box_hi, t.ncen);
        note_launch();
    }
}

int build_tree(Ctx* c, cudaStream_t s) {
    Tree& t = c->tree;
    const int64_t n = c->n;
    int rc = alloc_tree(c, std::max<int64_t>(1024, 2 * n / std::max(1, c->p.leaf_size) + 64), s);
    if (rc) return rc;
    int32_t* host = c->host_small + 8;   // kTreeLevels + 1 entries (the counters' place, unused here)
    static_assert(8 + kTreeLevels + 1 <= 64, "pinned scratch");
    for (;;) {
        if ((rc = launch_nodes(c, 1, nullptr, nullptr, nullptr, s))) return rc;
        cudaMemcpyAsync(host, t.level_cnt, (kTreeLevels + 1) * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
        if ((rc = check_cuda(cudaStreamSynchronize(s), "octree nodes"))) return rc;
        t.count = host[kTreeLevels];
        if (t.count <= t.cap) break;
        cudaMemsetAsync(c->err, 0, sizeof(unsigned), s);
        if ((rc = alloc_tree(c, t.count + t.count / 4, s))) return rc;
    }
    t.nlevels = 0;
    for (int l = 0; l < kTreeLevels; ++l)
        if (host[l] > 0) t.nlevels = l;
    t.nroots = 1;
    launch_up<true>(c, t.count, t.nlevels, s);
    cudaMemsetAsync(c->start_tab, 0xff, kStartTableSize * sizeof(int32_t), s);
    k_start_table<<<(int)std::min<int64_t>((t.count + 255) / 256, kTreeGrid), 256, 0, s>>>(
        t.level_cnt, t.cap, t.nlink, t.nlevel, c->pfix, nullptr, c->start_tab);
    note_launch();
    c->start_valid = true;
    return check_cuda(cudaGetLastError(), "octree build");
}

int refresh_hmax(Ctx* c, cudaStream_t s) {
    launch_up<false>(c, c->tree.count, c->tree.nlevels, s);
    return check_cuda(cudaGetLastError(), "hmax refresh");
}

// Forest of one octree per box (batch path).  Box k's particles are the ranks
// [box_off[k], box_off[k+1]) (sorted by box, then key); node k < nbox is box k's
// root.  Nothing is read back, so that the build can be captured in a CUDA graph.
int build_forest(Ctx* c, int nbox, const int64_t* box_off_dev, const int32_t* box_of_rank, int32_t* start_tabs,
                 cudaStream_t s, const int32_t* box_cfg) {
    Tree& t = c->tree;
    c->start_valid = false;   // the single-box table does not describe a forest
    t.count = t.cap;          // bounds
    t.nlevels = kKeyLevels;
    t.nroots = nbox;
    int rc = launch_nodes(c, nbox, box_off_dev, box_of_rank, box_cfg, s);
    if (rc) return rc;
    launch_up<true>(c, t.cap, kKeyLevels, s);
    if (start_tabs) {
        cudaMemsetAsync(start_tabs, 0xff, (size_t)nbox * kStartTableSize * sizeof(int32_t), s);
        k_start_table<<<kTreeGrid, 256, 0, s>>>(t.level_cnt, t.cap, t.nlink, t.nlevel, c->pfix, box_of_rank, start_tabs);
        note_launch();
    }
    return check_cuda(cudaGetLastError(), "forest build");
}

int gather_particles(Ctx* c, const double* pos, const float* m, cudaStream_t s) {
    k_gather<<<blocks_for(c->n, 256), 256, 0, s>>>(c->n, c->perm, pos, m, c->xd, c->yd, c->zd,
                                                  c->pfix, c->poff);
    note_launch();
    return check_cuda(cudaGetLastError(), "gather");
}

}  // namespace sphgrp
