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

__device__ __forceinline__ int key_digit(uint64_t key, int shift) { return (int)((key >> shift) & 7u); }

// Octant boundaries of the key range [lo, hi) (hi > lo) at the digit of `shift`: b[d] is
// the first index whose digit is >= d, b[0] = lo, b[8] = hi (digits are non-decreasing
// in the range).  The seven lower bounds run in lockstep: each step halves a range of
// the same length for all of them, so their loads are independent and a node's search
// costs the latency of one binary search, not of seven in a row.
__device__ __forceinline__ void octant_bounds(const uint64_t* __restrict__ keys, int lo, int hi, int shift,
                                              int (&b)[9]) {
    int base[7];
#pragma unroll
    for (int d = 0; d < 7; ++d) base[d] = lo;
    // invariant: indices below base[d] have digit < d + 1, and the bound lies in
    // [base[d], base[d] + n]
    int n = hi - lo;
    while (n > 1) {
        const int half = n >> 1;
        int dg[7];
#pragma unroll
        for (int d = 0; d < 7; ++d) dg[d] = key_digit(keys[base[d] + half], shift);
#pragma unroll
        for (int d = 0; d < 7; ++d)
            if (dg[d] < d + 1) base[d] += half;
        n -= half;
    }
    b[0] = lo;
    b[8] = hi;
#pragma unroll
    for (int d = 0; d < 7; ++d) b[d + 1] = base[d] + (key_digit(keys[base[d]], shift) < d + 1 ? 1 : 0);
}

// Cells of the top levels 1 .. kTopLevels: the first index of every non-empty cell, in a
// direct-indexed table per level (8^l entries at offset top_offset(l); -1 = empty).  A
// level-l node (l < kTopLevels) then reads its octant bounds from the 8 entries of its
// children instead of searching a key range of up to n keys, which at these levels is
// one long chain of dependent loads for a handful of threads.
constexpr int kTopLevels = 6;
constexpr int kTopTableSize = 299592;   // 8 + 8^2 + ... + 8^6
__host__ __device__ constexpr int top_offset(int l) { return ((1 << (3 * l)) - 8) / 7; }   // 8 + ... + 8^(l-1)
static_assert(top_offset(kTopLevels + 1) == kTopTableSize, "top-level cell table size");

// i starts a cell at every level deeper than the number of leading digits its key shares
// with key i - 1 (digit j of a 63-bit key is bits 62 - 3j .. 60 - 3j, so the first
// differing digit of x = k_i ^ k_{i-1} is (clz(x) - 1) / 3)
__global__ void k_top_cells(const uint64_t* __restrict__ keys, int64_t n, int32_t* __restrict__ tab) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t k = keys[i];
    int d = 0;
    if (i > 0) {
        const uint64_t x = k ^ keys[i - 1];
        d = x == 0 ? kKeyLevels : (__clzll((long long)x) - 1) / 3;
    }
    for (int l = d + 1; l <= kTopLevels; ++l) tab[top_offset(l) + (int)(k >> (3 * (kKeyLevels - l)))] = (int32_t)i;
}

// octant bounds of a node of level `level` over the keys [lo, hi): from the top-cell
// table above the top levels (tab non-null), else by the lockstep search
__device__ __forceinline__ void node_bounds(const uint64_t* __restrict__ keys, const int32_t* __restrict__ tab,
                                            int level, int lo, int hi, int (&b)[9]) {
    if (tab && level < kTopLevels) {
        const int P = level == 0 ? 0 : (int)(keys[lo] >> (3 * (kKeyLevels - level)));
        const int32_t* ch = tab + top_offset(level + 1) + 8 * P;
        int st[8];
#pragma unroll
        for (int d = 0; d < 8; ++d) st[d] = ch[d];
        b[8] = hi;
#pragma unroll
        for (int d = 7; d >= 0; --d) b[d] = st[d] >= 0 ? st[d] : b[d + 1];
        return;
    }
    octant_bounds(keys, lo, hi, 3 * (kKeyLevels - 1 - level), b);
}

// Octrees are built level by level over one or many boxes (a forest): the roots are nodes
// 0 .. nbox - 1, the nodes of a level are contiguous and so are a node's children, and the
// number of nodes of every level stays on the device (lcnt), so that the levels follow each
// other without a read-back.  Within a level the nodes' order varies from run to run (a
// block takes the ids of its nodes' children with one atomic); walks and results do not
// depend on it.

// first node and number of nodes of a level
__device__ __forceinline__ void level_range(const int32_t* __restrict__ lcnt, int level, int64_t cap, int& a, int& nf) {
    int64_t first = 0;
    for (int l = 0; l < level; ++l) first += lcnt[l];
    a = (int)min(first, cap);
    nf = (int)max((int64_t)0, min((int64_t)lcnt[level], cap - first));
}

__global__ void k_tree_roots(int nbox, const int64_t* __restrict__ box_off, int64_t n, int4* __restrict__ nlink,
                             float4* __restrict__ next, int32_t* __restrict__ nlevel, int32_t* __restrict__ nparent,
                             uint32_t* __restrict__ narrive, int32_t* __restrict__ lcnt) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < nbox) {
        const int64_t lo = box_off ? box_off[k] : 0, hi = box_off ? box_off[k + 1] : n;
        nlink[k] = make_int4((int)lo, (int)(hi - lo), -1, -1);
        next[k] = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0));
        nlevel[k] = 0;
        nparent[k] = -1;
        narrive[k] = 0u;
    }
    if (k < kTreeLevels) lcnt[k] = k == 0 ? nbox : 0;
}

// The nodes of one level with more than leaf_size particles get their children, one per
// non-empty octant.  box_cfg (optional): per box, bits 16..23 = that box's leaf size (0:
// leaf_size); the node's box is the box of its first particle.  Children beyond the
// capacity are not created: their parent stays a leaf, the ids it was given below the
// capacity become empty leaves that nothing links to, and the error flag is set.
__global__ void __launch_bounds__(256) k_split_level(const uint64_t* __restrict__ keys, int4* __restrict__ nlink,
                                                     float4* __restrict__ next, int32_t* __restrict__ nlevel,
                                                     int32_t* __restrict__ nparent, uint32_t* __restrict__ narrive,
                                                     int32_t* __restrict__ lcnt, int level, int leaf_size,
                                                     const int32_t* __restrict__ tab,
                                                     const int32_t* __restrict__ box_cfg,
                                                     const int32_t* __restrict__ box_of_rank, int64_t cap,
                                                     unsigned* err) {
    __shared__ int wtot[8];
    __shared__ int first;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int a, nf;
    level_range(lcnt, level, cap, a, nf);
    for (int k0 = blockIdx.x * 256; k0 < nf; k0 += gridDim.x * 256) {   // block-uniform
        const int k = k0 + threadIdx.x;
        int4 L = make_int4(0, 0, -1, -1);
        int bd[9];
        int nc = 0;
        if (k < nf) {
            L = nlink[a + k];
            int leaf = leaf_size;
            if (box_cfg && L.y > 0) {
                const int lb = (box_cfg[box_of_rank[L.x]] >> 16) & 0xff;
                if (lb > 0) leaf = lb;
            }
            if (L.y > leaf && level < kKeyLevels) {
                node_bounds(keys, tab, level, L.x, L.x + L.y, bd);
#pragma unroll
                for (int d = 0; d < 8; ++d) nc += bd[d + 1] > bd[d] ? 1 : 0;
            }
        }
        int inc = nc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) wtot[w] = inc;
        __syncthreads();
        int pre = inc - nc, tot = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (q < w) pre += wtot[q];
            tot += wtot[q];
        }
        if (threadIdx.x == 0 && tot > 0) first = atomicAdd(&lcnt[level + 1], tot);
        __syncthreads();
        if (nc > 0) {
            const int64_t child0 = (int64_t)a + nf + first + pre;
            if (child0 + nc > cap) {
                atomicOr(err, kErrNodes);
                for (int64_t id = child0; id < min(child0 + nc, cap); ++id) {   // counted: empty leaves
                    nlink[id] = make_int4(0, 0, -1, -1);
                    next[id] = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0));
                    nlevel[id] = level + 1;
                    nparent[id] = -1;
                    narrive[id] = 0u;
                }
            } else {
                int c = 0;
#pragma unroll
                for (int d = 0; d < 8; ++d) {
                    if (bd[d + 1] > bd[d]) {
                        const int id = (int)child0 + c;
                        nlink[id] = make_int4(bd[d], bd[d + 1] - bd[d], -1, c + 1 < nc ? id + 1 : L.w);
                        next[id] = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0));
                        nlevel[id] = level + 1;
                        nparent[id] = a + k;
                        narrive[id] = 0u;
                        ++c;
                    }
                }
                next[a + k].w = __int_as_float(nc);
                L.z = (int)child0;
                nlink[a + k] = L;
            }
        }
        __syncthreads();   // wtot and first are rewritten by the next round
    }
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

// Node arrays for cap nodes (the old contents are dropped).
int alloc_tree(Ctx* c, int64_t cap) {
    Tree& t = c->tree;
    if (!t.level_cnt && cudaMalloc(&t.level_cnt, kTreeLevels * sizeof(int32_t)) != cudaSuccess) {
        t.level_cnt = nullptr;
        cudaGetLastError();
        return set_error(SPHGRP_ENOMEM, "octree level counts");
    }
    if (cap <= t.cap) return SPHGRP_OK;
    void** ptrs[] = {(void**)&t.ncen, (void**)&t.next, (void**)&t.nlink, (void**)&t.nlevel, (void**)&t.nparent,
                     (void**)&t.narrive, (void**)&t.box_lo, (void**)&t.box_hi};
    const size_t bytes[] = {sizeof(uint4), sizeof(float4), sizeof(int4), sizeof(int32_t), sizeof(int32_t),
                            sizeof(uint32_t), sizeof(uint4), sizeof(uint4)};
    for (void** p : ptrs) {
        if (*p) cudaFree(*p);
        *p = nullptr;
    }
    t.cap = 0;
    for (int k = 0; k < 8; ++k) {
        if (cudaMalloc(ptrs[k], (size_t)cap * bytes[k]) != cudaSuccess) {
            cudaGetLastError();
            return set_error(SPHGRP_ENOMEM, "octree allocation failed");
        }
    }
    t.cap = cap;
    return SPHGRP_OK;
}

static void launch_levels(Ctx* c, int from, int to, int nbox, const int32_t* tab, const int32_t* box_cfg,
                          const int32_t* box_of_rank, cudaStream_t s) {
    Tree& t = c->tree;
    for (int level = from; level < to; ++level) {
        // at most 8^level nodes per box
        const int64_t bound = level < 7 ? std::min<int64_t>(t.cap, (int64_t)nbox << (3 * level)) : t.cap;
        const int grid = (int)std::min<int64_t>((bound + 255) / 256, kTreeGrid);
        k_split_level<<<grid, 256, 0, s>>>(c->keys, t.nlink, t.next, t.nlevel, t.nparent, t.narrive, t.level_cnt, level,
                                           c->p.leaf_size, tab, box_cfg, box_of_rank, t.cap, c->err);
        note_launch();
    }
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
    int rc = alloc_tree(c, std::max<int64_t>(1024, 2 * n / std::max(1, c->p.leaf_size) + 64));
    if (rc) return rc;
    if (!t.top_cells && cudaMalloc(&t.top_cells, kTopTableSize * sizeof(int32_t)) != cudaSuccess) {
        t.top_cells = nullptr;
        return set_error(SPHGRP_ENOMEM, "octree top-cell table");
    }
    int32_t* top = t.top_cells;
    cudaMemsetAsync(top, 0xff, kTopTableSize * sizeof(int32_t), s);
    k_top_cells<<<blocks_for(n, 256), 256, 0, s>>>(c->keys, n, top);
    note_launch();
    int32_t* host = c->host_small + 8;   // kTreeLevels entries (the counters' place, unused here)
    static_assert(8 + kTreeLevels <= 64, "pinned scratch");
    for (;;) {
        k_tree_roots<<<1, 256, 0, s>>>(1, nullptr, n, t.nlink, t.next, t.nlevel, t.nparent, t.narrive, t.level_cnt);
        note_launch();
        // as many levels as the last build had and two more; the rest if they were too few
        int upto = std::min(kKeyLevels, t.nlevels + 2);
        launch_levels(c, 0, upto, 1, top, nullptr, nullptr, s);
        cudaMemcpyAsync(host, t.level_cnt, kTreeLevels * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
        if ((rc = check_cuda(cudaStreamSynchronize(s), "octree levels"))) return rc;
        while (upto < kKeyLevels && host[upto] > 0) {
            launch_levels(c, upto, kKeyLevels, 1, top, nullptr, nullptr, s);
            upto = kKeyLevels;
            cudaMemcpyAsync(host, t.level_cnt, kTreeLevels * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
            if ((rc = check_cuda(cudaStreamSynchronize(s), "octree levels"))) return rc;
        }
        int64_t total = 0;
        t.nlevels = 0;
        for (int l = 0; l < kTreeLevels; ++l) {
            total += host[l];
            if (host[l] > 0) t.nlevels = l;
        }
        t.count = total;
        if (total <= t.cap) break;
        // too few nodes: the counts of the deeper levels are those of the children that
        // would have been made up to there
        cudaMemsetAsync(c->err, 0, sizeof(unsigned), s);
        if ((rc = alloc_tree(c, std::max(total + total / 2, 2 * t.cap)))) return rc;
    }
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
    k_tree_roots<<<blocks_for(std::max(nbox, kTreeLevels), 256), 256, 0, s>>>(
        nbox, box_off_dev, c->n, t.nlink, t.next, t.nlevel, t.nparent, t.narrive, t.level_cnt);
    note_launch();
    launch_levels(c, 0, kKeyLevels, nbox, nullptr, box_cfg, box_of_rank, s);
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
