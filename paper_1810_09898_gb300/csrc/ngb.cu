// Neighbour search and the SPH loops that consume it, forward and backward.
//
// Two forms (Sec. 1.1 standard search, Sec. 2.1 Neighbour Recycling):
//  * individual: every active particle is searched by itself, a warp walking the octree
//    for its sphere of radius h_i (hydro: max(h_i, node hmax)): a group of one member.
//    The calls that export neighbour lists walk with a thread per particle, depth-first
//    by skip pointers;
//  * grouped: one warp per group of consecutive active particles (key order).  The
//    warp walks the octree cooperatively once for the group (32 nodes tested per
//    step) over the members' box dilated by their largest radius, takes the particles
//    of the opened nodes (the common superset) 32 at a time, keeps those inside the
//    dilated box in a shared-memory tile, and every member filters the tile down to
//    its own neighbours.
//
// The grouped kernel is shared by four kinds of pair loop: density (0), hydro (1),
// and the adjoints of the hydro accelerations (2) and of the density (3); the two
// adjoints recompute their pair terms over the same grouped candidate tiles instead
// of storing pair lists.
//
// Pair decisions are taken in FP32 on coordinates relative to a fixed-point centre;
// pairs whose FP32 r^2 falls inside the proven error band around the threshold are
// re-decided from the FP64 positions with the oracle's exact arithmetic, so the
// neighbour sets are those of the FP64 definition.  Sums are FP32 (forward sums
// compensated across tiles).
#include "search_args.cuh"

namespace sphgrp {

constexpr int kWarpsPerBlock = 4;
constexpr int kStackCap = kStackSharedMax;     // walk stack entries in shared memory
constexpr int kRangeCap = 64;                  // pending particle ranges (ring, power of two)
constexpr int kSpillCap = kStackSpillPerWarp;  // overflow entries per warp (global memory)
// candidates of a tile: density kinds, and those whose candidates carry records (larger
// tiles balance the lanes of phase B better, until fewer warps fit)
constexpr int kTileD = 160;
constexpr int kTileR = 128;
constexpr int kPartMax = 32;                   // members searched at once (one per lane)
// The walk takes a node of at most this many particles whole instead of opening it.
constexpr int kWalkWhole = 32;
// A single member's region is smaller (1.0M clustered particles one by one, density + hydro:
// 9.62 ms at 32, 9.47 at 16 and at 8, 9.85 at 48).
constexpr int kWalkWholeSingle = 16;


// per-lane counts of one launch, summed in 64 bits
struct LocalCounters {
    unsigned tests = 0, pairs = 0, retests = 0;
};
// counts of a warp's walks, in its shared memory (they would hold registers through every
// search)
struct WalkCounters {
    unsigned walks, nodes, cands, deep;
};

__device__ __forceinline__ unsigned long long warp_sum(unsigned v) {
    unsigned long long t = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

__device__ __forceinline__ void flush_counters(const SearchArgs& a, const LocalCounters& lc, const WalkCounters& wc,
                                               int lane) {
    // warp-reduce then one atomic per warp
    const unsigned long long tests = warp_sum(lc.tests), pairs = warp_sum(lc.pairs), retests = warp_sum(lc.retests);
    if (lane == 0) {
        if (wc.walks) atomicAdd(&a.ctr->walks, (unsigned long long)wc.walks);
        if (wc.nodes) atomicAdd(&a.ctr->nodes, (unsigned long long)wc.nodes);
        if (wc.cands) atomicAdd(&a.ctr->cands, (unsigned long long)wc.cands);
        if (tests) atomicAdd(&a.ctr->tests, tests);
        if (pairs) atomicAdd(&a.ctr->pairs, pairs);
        if (retests) atomicAdd(&a.ctr->retests, retests);
        atomicMax(&a.ctr->max_stack, (unsigned long long)wc.deep);
    }
}

// largest of the lanes' non-negative floats
__device__ __forceinline__ float warp_max(float v) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// Squared distance, in fixed-point units^2 and rounded down, from the point C to a
// node's box (conservative: never larger than the true distance).
__device__ __forceinline__ float node_gap2(const uint4& cen, const float4& ext, uint32_t cx,
                                           uint32_t cy, uint32_t cz) {
    float dx = fabsf(__int2float_rz((int32_t)(cen.x - cx)));
    float dy = fabsf(__int2float_rz((int32_t)(cen.y - cy)));
    float dz = fabsf(__int2float_rz((int32_t)(cen.z - cz)));
    float gx = fmaxf(__fsub_rd(dx, ext.x), 0.0f);
    float gy = fmaxf(__fsub_rd(dy, ext.y), 0.0f);
    float gz = fmaxf(__fsub_rd(dz, ext.z), 0.0f);
    return __fadd_rd(__fadd_rd(__fmul_rd(gx, gx), __fmul_rd(gy, gy)), __fmul_rd(gz, gz));
}

// radius in box units -> squared radius in fixed-point units, rounded up, with a
// relative margin for the FP32 error of the radius itself
__device__ __forceinline__ float radius2_units(float r_box) {
    float r = __fmul_ru(__fmul_ru(r_box, 1.0000010f), 4294967296.0f);
    return __fmul_ru(r, r);
}

// Members farther than this many smoothing lengths from the group centre (per axis)
// evaluate the pair physics from exact fixed-point differences: the FP32 difference of
// two centre-relative coordinates loses up to |m| / h ulps of r, so below this reach the
// pair terms carry at most about 8 ulps (1e-6 relative) of error, far inside the density
// (1e-5) and acceleration (1e-4) bars; the decisions are exact at any reach (the band's
// |m|^2 term).  The exact path reloads both fixed-point records from global memory.
constexpr float kPreciseReach = 8.0f;

// x_j - x_k from the fixed-point layout: exact integer minimum image plus the offsets.
__device__ __forceinline__ float fix_diff(uint32_t Xj, float oj, uint32_t Xk, float ok) {
    return (__int2float_rn((int32_t)(Xj - Xk)) + (oj - ok)) * kUnitToBox;
}

// Difference of two coordinates relative to one centre.  Both lie in [-1/2, 1/2); when
// a group can reach half the box (WRAP) the difference is brought back to the nearest
// periodic image, otherwise it already is that image (|m| + h < 1/2 for every member).
template <bool WRAP>
__device__ __forceinline__ float rel_diff(float p, float m) {
    float d = p - m;
    if (WRAP) d -= rintf(d);
    return d;
}

// dW/dr = kSkernel h^-4 dw/dq for the M4 spline W = 8 / (pi h^3) w(r / h)
constexpr float kSkernel = 2.54647908947032537f;   // 8 / pi

// hardware reciprocal square root and reciprocal (1 ulp; arguments of normal size: a
// subnormal one is flushed to zero and gives infinity)
__device__ __forceinline__ float rsqrt_fast(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// the same, subnormal arguments included (three more instructions)
__device__ __forceinline__ float rsqrt_any(float x) {
    float y;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Least r^2 of normal size: a pair closer than its root, 1.1e-19 of the box, is taken as
// coincident where its terms vanish with r (kernel gradients; the viscosity's with a
// softening eps > 0); the hydro adjoint, whose derivative of the pair force does not, takes
// its root by rsqrt_any.  Hydro of 4.2M 6.46 ms with and without; subnormal roots everywhere
// cost it 1.3% and backward of 2.1M 1.1%, in the adjoint alone 0.5% (9.72 -> 9.77 ms).
constexpr float kMinR2 = 1.17549435e-38f;
__device__ __forceinline__ float rcp_fast(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// q = r / h rounded on its own: fused into the 1 - q of the splines it would differ by an
// ulp between kernels that inline the same pair terms
__device__ __forceinline__ float q_of(float r, float hinv) { return __fmul_rn(r, hinv); }

// M4 slope w'(q) (zero for q >= 1; q >= 0)
__device__ __forceinline__ float m4_slope(float q) {
    const float u = __saturatef(1.0f - q);
    return q <= 0.5f ? q * fmaf(18.0f, q, -12.0f) : -6.0f * u * u;
}

// w(q) and 3 w + q w' of the M4 spline (zero for q >= 1; q >= 0): inside 1/2
// 1 + q^2 (6q - 6) and 3 + q^2 (36q - 30), outside 2 u^3 and 6 u^2 (1 - 2q), u = 1 - q
__device__ __forceinline__ void m4_density(float q, float& w, float& v) {
    const float u = __saturatef(1.0f - q);
    const float q2 = q * q, u2 = u * u;
    const bool inner = q <= 0.5f;
    w = inner ? fmaf(q2, fmaf(6.0f, q, -6.0f), 1.0f) : 2.0f * u2 * u;
    v = inner ? fmaf(q2, fmaf(36.0f, q, -30.0f), 3.0f) : 6.0f * u2 * fmaf(-2.0f, q, 1.0f);
}

// M4 shape w(q), w'(q), w''(q) (zero for q >= 1)
__device__ __forceinline__ void m4_shape2(float q, float& w, float& dw, float& d2w) {
    float u = 1.0f - q;
    bool inner = q <= 0.5f;
    w = inner ? fmaf(q * q, 6.0f * q - 6.0f, 1.0f) : 2.0f * u * u * u;
    dw = inner ? q * (18.0f * q - 12.0f) : -6.0f * u * u;
    d2w = inner ? fmaf(36.0f, q, -12.0f) : 12.0f * u;
    if (q >= 1.0f) { w = 0.0f; dw = 0.0f; d2w = 0.0f; }
}

// ---------------------------------------------------------------------------------
// Asynchronous 16-byte copies global -> shared (both addresses 16-byte aligned)
// ---------------------------------------------------------------------------------

__device__ __forceinline__ void copy16_async(float4* dst, const float4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// packed FP32 pairs (two FMAs in one issue slot)
__device__ __forceinline__ unsigned long long pair_of(float lo, float hi) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ unsigned long long fma_pair(unsigned long long a, unsigned long long b,
                                                       unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long add_pair(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// m shifted left by one, the sign of v entering at the bottom
__device__ __forceinline__ uint32_t push_sign(uint32_t m, uint32_t v) { return __funnelshift_l(v, m, 1); }

__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---------------------------------------------------------------------------------
// Per-member state of the four pair loops
// ---------------------------------------------------------------------------------

// position part shared by all members: coordinates relative to the group centre (the
// exact fixed-point position is reloaded by the rare paths that need it)
// Lower decision threshold of members whose physics takes exact differences: no pair lies
// below it, so every one goes through the decision's slow path (one-sided kinds: h2lo;
// symmetric ones: -bk).
constexpr float kAlwaysSlow = -3.0e38f;

struct MemberPos {
    float mx, my, mz;
    int rank;           // -1: slot empty
    int n;              // neighbours found
    int64_t xpos;       // export write position
};

// a member's key-ordered records, loaded once per search (rank < 0: an empty slot)
struct MemberRec {
    int rank;
    uint4 P;
    float4 O;
    double h;
};

__device__ __forceinline__ MemberRec load_member(const SearchArgs& a, int rank) {
    MemberRec r;
    r.rank = rank;
    r.P = make_uint4(0u, 0u, 0u, 0u);
    r.O = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    r.h = 1.0;
    if (rank >= 0) {
        r.P = a.pfix[rank];
        r.O = a.poff[rank];
        r.h = a.h64[rank];
    }
    return r;
}

// precise: far from the group centre, physics from exact differences
__device__ __forceinline__ bool pos_init(MemberPos& M, const MemberRec& rec, uint32_t cx, uint32_t cy, uint32_t cz,
                                         float hf, bool& precise) {
    const int rank = rec.rank;
    M.rank = rank;
    M.n = 0;
    M.xpos = 0;
    precise = false;
    if (rank < 0) {
        M.mx = M.my = M.mz = 0.0f;
        return false;
    }
    M.mx = rel_coord(rec.P.x, rec.O.x, cx);
    M.my = rel_coord(rec.P.y, rec.O.y, cy);
    M.mz = rel_coord(rec.P.z, rec.O.z, cz);
    precise = fmaxf(fabsf(M.mx), fmaxf(fabsf(M.my), fabsf(M.mz))) > kPreciseReach * hf;
    return true;
}

// density member
struct DMember : MemberPos {
    float hinv;
    float h2lo, h2hi;   // decided-inside below h2lo, candidate below h2hi
    float thr_dot;      // phase-A threshold of |p|^2 - 2 p.m (= h2hi - |m|^2)
    float s0, c0, s1, c1;   // compensated totals: sum m w, sum m (3w + q w')
    float p0, p1;           // plain partial sums of the current tile
};

// density member with the second derivative (backward): also the sum of the W_hh shape
struct D2Member : DMember {
    float s2, c2, p2;
};

// density member with the velocity derivatives over the same density set: the sums of
// -m v_ij . grad W (divergence) and m v_ij x grad W (curl) at h_i, before the 1/rho
struct DVMember : DMember {
    float vx, vy, vz, sk;
    float sd, cd, sx, cx_, sy, cy_, sz, cz_;   // compensated totals
    float pd, px_, py_, pz_;                   // plain partial sums of the current tile
};

// density member of the recycled smoothing-length iteration: besides the sums at h it
// keeps every candidate inside the widened radius h_w in its slice's sub-list
struct DLMember : DMember {
    float hwf;          // h_w (FP32): the walk radius covers it
    float h2whi;        // widened candidate threshold of the difference form
    float thr_dot_w;    // widened phase-A threshold of the dot form
    int lsub;           // capacity of this lane's sub-list
    int lcnt;           // candidates found (above lsub: the sub-list overflowed)
    int32_t* lptr;      // this lane's sub-list
};

// members of the symmetric criterion |r| < max(h_i, h_j) (hydro and both adjoints)
struct SymMember : MemberPos {
    float h, hinv, sk;  // sk = 8 / (pi h^4): dW/dr = sk * dw/dq
    float h2, bk;       // h^2 (FP32 of the FP64 square), band offset 8 b |m|^2
    float bk_dot;       // bk - |m|^2: phase-A offset of the dot form
};

struct HMember : SymMember {
    float vx, vy, vz, cs, A;
    float rho4, fb4;   // a quarter of the density and of the viscosity limiter (1 without one)
    float sx, cx_, sy, cy_, sz, cz_, su, cu;   // compensated totals
    float px_, py_, pz_, pu;                   // plain partial sums of the current tile
};

// hydro-adjoint member: the forward hydro state, the weights w_k = dL/da_k, and the
// adjoint sums of x, v, m, h, rho and A = f P / rho^2
struct HAMember : SymMember {
    float vx, vy, vz, cs, A, rho4, m;   // rho4: a quarter of the density
    float wx, wy, wz;
    float xb[3], vb[3], mb, hb, rb, Ab;
};

// density-adjoint member: the coefficients alpha = adjoint of rho at fixed h (with the
// implicit-h term) and beta = adjoint of dRho/dh
struct DAMember : SymMember {
    float alpha, beta, m;
    float xb[3], mb;
};

// velocity-derivative member (density criterion): sums of -m v_ij . grad W (divergence)
// and m v_ij x grad W (curl), v_ij = v_i - v_j, grad W at h_i
struct VMember : MemberPos {
    float hinv;
    float h2lo, h2hi;
    float thr_dot;
    float sk;               // 8 / (pi h^4): dW/dr = sk * dw/dq
    float vx, vy, vz;
    float rrho;             // 1 / rho_i
    float sd, cd, sx, cx_, sy, cy_, sz, cz_;   // compensated totals
    float pd, px_, py_, pz_;                   // plain partial sums of the current tile
};

__device__ __forceinline__ void member_init(DMember& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    M.s0 = M.c0 = M.s1 = M.c1 = 0.0f;
    M.p0 = M.p1 = 0.0f;
    const double h = rec.h;
    float hf = (float)h;
    bool precise;
    if (!pos_init(M, rec, cx, cy, cz, hf, precise)) {
        M.hinv = 0.0f;
        M.h2lo = M.h2hi = -1.0f;
        M.thr_dot = -3.0e38f;
        return;
    }
    M.hinv = 1.0f / hf;
    float h2 = (float)(h * h);
    float m2 = M.mx * M.mx + M.my * M.my + M.mz * M.mz;
    float bk = 8.0f * kBandRel * m2;
    M.h2hi = fmaf(h2, 1.0f + 3.0f * kBandRel, bk);
    M.h2lo = precise ? kAlwaysSlow : fmaf(h2, 1.0f - 3.0f * kBandRel, -bk);
    M.thr_dot = M.h2hi - m2;
}

__device__ __forceinline__ void member_init(D2Member& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    member_init(static_cast<DMember&>(M), a, rec, cx, cy, cz);
    M.s2 = M.c2 = M.p2 = 0.0f;
}

__device__ __forceinline__ void member_init(DVMember& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    member_init(static_cast<DMember&>(M), a, rec, cx, cy, cz);
    M.sd = M.cd = M.sx = M.cx_ = M.sy = M.cy_ = M.sz = M.cz_ = 0.0f;
    M.pd = M.px_ = M.py_ = M.pz_ = 0.0f;
    M.vx = M.vy = M.vz = M.sk = 0.0f;
    if (rec.rank < 0) return;
    const float4 V = a.hyd0[rec.rank];
    M.vx = V.x;
    M.vy = V.y;
    M.vz = V.z;
    M.sk = kSkernel * (M.hinv * M.hinv) * (M.hinv * M.hinv);
}

__device__ __forceinline__ void member_init(DLMember& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    member_init(static_cast<DMember&>(M), a, rec, cx, cy, cz);
    M.lsub = 0;
    M.lcnt = 0;
    M.lptr = nullptr;
    if (rec.rank < 0) {
        M.hwf = 0.0f;
        M.h2whi = -1.0f;
        M.thr_dot_w = -3.0e38f;
        return;
    }
    // the same band as the thresholds at h, at h_w: every candidate with an exact
    // distance below h_w passes it
    const double hw = rec.h * a.list_widen;
    M.hwf = (float)hw;
    const float m2 = M.mx * M.mx + M.my * M.my + M.mz * M.mz;
    M.h2whi = fmaf((float)(hw * hw), 1.0f + 3.0f * kBandRel, 8.0f * kBandRel * m2);
    M.thr_dot_w = M.h2whi - m2;
}

__device__ __forceinline__ bool sym_init(SymMember& M, const MemberRec& rec, uint32_t cx, uint32_t cy,
                                         uint32_t cz) {
    const double h = rec.h;
    M.h = (float)h;
    bool precise;
    if (!pos_init(M, rec, cx, cy, cz, M.h, precise)) {
        M.h = 0.0f; M.hinv = 0.0f; M.sk = 0.0f;
        M.h2 = -1.0f; M.bk = -1.0f;
        M.bk_dot = -3.0e38f;
        return false;
    }
    M.h2 = (float)(h * h);
    float m2 = M.mx * M.mx + M.my * M.my + M.mz * M.mz;
    M.bk = precise ? -kAlwaysSlow : 8.0f * kBandRel * m2;
    M.bk_dot = 8.0f * kBandRel * m2 - m2;
    return true;
}

__device__ __forceinline__ void member_init(HMember& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    M.sx = M.cx_ = M.sy = M.cy_ = M.sz = M.cz_ = M.su = M.cu = 0.0f;
    M.px_ = M.py_ = M.pz_ = M.pu = 0.0f;
    M.vx = M.vy = M.vz = M.cs = M.A = M.rho4 = 0.0f;
    M.fb4 = 0.25f;
    if (!sym_init(M, rec, cx, cy, cz)) return;
    float4 H0 = a.hyd0[rec.rank];
    float4 H1 = a.hyd1[rec.rank];   // {A, rho / 4, 1/h, limiter / 4}
    M.hinv = H1.z;
    M.sk = kSkernel * (H1.z * H1.z) * (H1.z * H1.z);
    M.fb4 = H1.w;
    M.vx = H0.x; M.vy = H0.y; M.vz = H0.z; M.cs = H0.w;
    M.A = H1.x;
    M.rho4 = H1.y;
}

__device__ __forceinline__ void member_init(HAMember& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    for (int k = 0; k < 3; ++k) M.xb[k] = M.vb[k] = 0.0f;
    M.mb = M.hb = M.rb = M.Ab = 0.0f;
    M.vx = M.vy = M.vz = M.cs = M.A = M.rho4 = M.m = 0.0f;
    M.wx = M.wy = M.wz = 0.0f;
    if (!sym_init(M, rec, cx, cy, cz)) return;
    float4 H0 = a.hyd0[rec.rank];
    float4 H1 = a.hyd1[rec.rank];
    float4 Wt = a.wadj[rec.rank];
    M.hinv = H1.z;
    M.sk = H1.w;
    M.vx = H0.x; M.vy = H0.y; M.vz = H0.z; M.cs = H0.w;
    M.A = H1.x;
    M.rho4 = H1.y;
    M.m = rec.O.w;
    M.wx = Wt.x; M.wy = Wt.y; M.wz = Wt.z;
}

__device__ __forceinline__ void member_init(DAMember& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    for (int k = 0; k < 3; ++k) M.xb[k] = 0.0f;
    M.mb = 0.0f;
    M.alpha = M.beta = M.m = 0.0f;
    if (!sym_init(M, rec, cx, cy, cz)) return;
    float4 D = a.dadj[rec.rank];
    M.alpha = D.x;
    M.beta = D.y;
    M.hinv = D.z;
    M.sk = D.w;
    M.m = rec.O.w;
}

__device__ __forceinline__ void member_init(VMember& M, const SearchArgs& a, const MemberRec& rec, uint32_t cx,
                                            uint32_t cy, uint32_t cz) {
    M.sd = M.cd = M.sx = M.cx_ = M.sy = M.cy_ = M.sz = M.cz_ = 0.0f;
    M.pd = M.px_ = M.py_ = M.pz_ = 0.0f;
    M.vx = M.vy = M.vz = 0.0f;
    M.sk = 0.0f;
    M.rrho = 0.0f;
    const double h = rec.h;
    float hf = (float)h;
    bool precise;
    if (!pos_init(M, rec, cx, cy, cz, hf, precise)) {
        M.hinv = 0.0f;
        M.h2lo = M.h2hi = -1.0f;
        M.thr_dot = -3.0e38f;
        return;
    }
    M.hinv = 1.0f / hf;
    float h2 = (float)(h * h);
    float m2 = M.mx * M.mx + M.my * M.my + M.mz * M.mz;
    float bk = 8.0f * kBandRel * m2;
    M.h2hi = fmaf(h2, 1.0f + 3.0f * kBandRel, bk);
    M.h2lo = precise ? kAlwaysSlow : fmaf(h2, 1.0f - 3.0f * kBandRel, -bk);
    M.thr_dot = M.h2hi - m2;
    const float4 H0 = a.hyd0[rec.rank];
    const float4 H1 = a.hyd1[rec.rank];
    M.vx = H0.x; M.vy = H0.y; M.vz = H0.z;
    M.rrho = 1.0f / H1.y;
    M.sk = H1.w;
}

// radius of the search sphere around a member (symmetric kinds: its own h; a node or a
// candidate widens it by its own)
__device__ __forceinline__ float member_radius(const DMember& M) { return M.rank < 0 ? 0.0f : 1.0f / M.hinv; }
__device__ __forceinline__ float member_radius(const DLMember& M) { return M.rank < 0 ? 0.0f : M.hwf; }
__device__ __forceinline__ float member_radius(const VMember& M) { return M.rank < 0 ? 0.0f : 1.0f / M.hinv; }
__device__ __forceinline__ float member_radius(const SymMember& M) { return M.rank < 0 ? 0.0f : M.h; }

// ---------------------------------------------------------------------------------
// Candidate tiles in shared memory: the candidates of a group that passed the test
// against its dilated box, in walk order, as FP32 coordinates relative to the group
// centre (w = |p|^2), with their mass (symmetric kinds: and h^2), rank and the kind's own
// records.  With S slices, the candidates go to the slices in turn, four at a time, and a
// slice's are contiguous (`rows` quads of them), so that phase A reads them by whole
// quads at constant strides and phase B finds a candidate by adding its number to the
// slice's start.  Phase A may read one row past the last (the next slice's or array's
// values) and drops its bits.
// ---------------------------------------------------------------------------------

template <int N>
struct alignas(16) PlainTileOf {
    static constexpr int cap = N;
    float x[N], y[N], z[N], w[N];
    float m[N];
    int r[N];           // ranks
    uint32_t masks[N];  // phase-A bit masks [word][lane]
};
using PlainTile = PlainTileOf<kTileD>;
struct SymTile : PlainTileOf<kTileR> {
    float h2[kTileR];       // h_j^2
};
struct VelTile : PlainTileOf<kTileR> {
    float4 v[kTileR];       // hyd0 {vx, vy, vz, -}
};
struct HydroTile : SymTile {
    float4 v[kTileR];       // hyd0 {vx, vy, vz, c}
    float4 h[kTileR];       // hyd1 {A, rho / 4, 1/h, limiter / 4}
};
struct HAdjTile : SymTile {
    float4 v[kTileR];       // hyd0 {vx, vy, vz, c}
    float4 h[kTileR];       // hyd1 {A, rho / 4, 1/h, 8/(pi h^4)}
    float4 wt[kTileR];      // wadj {wx, wy, wz, -}
};
struct DAdjTile : SymTile {
    float4 d[kTileR];       // dadj {alpha, beta, 1/h, 8/(pi h^4)}
};

// kind policies; min_blocks: resident blocks per SM (register budget; 0: compiler's choice)
struct KDens {
    static constexpr int min_blocks = 8;
    static constexpr int id = 0;
    static constexpr bool sym = false;
    using Member = DMember;
    using Tile = PlainTile;
};
struct KDens2 {
    static constexpr int min_blocks = 7;
    static constexpr int id = kKindDensity;
    static constexpr bool sym = false;
    using Member = D2Member;
    using Tile = PlainTile;
};
struct KDensVel {
    static constexpr int min_blocks = 5;
    static constexpr int id = kKindDensityVel;
    static constexpr bool sym = false;
    using Member = DVMember;
    using Tile = VelTile;
};
struct KDensList {
    static constexpr int min_blocks = 7;
    static constexpr int id = kKindDensityList;
    static constexpr bool sym = false;
    using Member = DLMember;
    using Tile = PlainTile;
};
struct KHydro {
    static constexpr int min_blocks = 5;
    static constexpr int id = 1;
    static constexpr bool sym = true;
    using Member = HMember;
    using Tile = HydroTile;
};
struct KHAdj {
    static constexpr int min_blocks = 4;
    static constexpr int id = 2;
    static constexpr bool sym = true;
    using Member = HAMember;
    using Tile = HAdjTile;
};
struct KDAdj {
    static constexpr int min_blocks = 6;
    static constexpr int id = 3;
    static constexpr bool sym = true;
    using Member = DAMember;
    using Tile = DAdjTile;
};
struct KVel {
    static constexpr int min_blocks = 0;
    static constexpr int id = 4;
    static constexpr bool sym = false;
    using Member = VMember;
    using Tile = VelTile;
};

// the kind's own records of a candidate that entered the tile at position t
__device__ __forceinline__ void stage_records(PlainTile&, const SearchArgs&, int, int) {}
__device__ __forceinline__ void stage_records(VelTile& T, const SearchArgs& a, int t, int rank) {
    copy16_async(&T.v[t], a.hyd0 + rank);
}
__device__ __forceinline__ void stage_records(HydroTile& T, const SearchArgs& a, int t, int rank) {
    copy16_async(&T.v[t], a.hyd0 + rank);
    copy16_async(&T.h[t], a.hyd1 + rank);
}
__device__ __forceinline__ void stage_records(HAdjTile& T, const SearchArgs& a, int t, int rank) {
    copy16_async(&T.v[t], a.hyd0 + rank);
    copy16_async(&T.h[t], a.hyd1 + rank);
    copy16_async(&T.wt[t], a.wadj + rank);
}
__device__ __forceinline__ void stage_records(DAdjTile& T, const SearchArgs& a, int t, int rank) {
    copy16_async(&T.d[t], a.dadj + rank);
}

// ---------------------------------------------------------------------------------
// Pair physics
// ---------------------------------------------------------------------------------

// Plain per-tile partial sums are folded into the compensated totals after every
// tile (or leaf): a few tens of terms in plain FP32, Kahan across blocks.
__device__ __forceinline__ void flush(DMember& M) {
    kahan_add(M.s0, M.c0, M.p0);
    kahan_add(M.s1, M.c1, M.p1);
    M.p0 = M.p1 = 0.0f;
}

__device__ __forceinline__ void flush(D2Member& M) {
    flush(static_cast<DMember&>(M));
    kahan_add(M.s2, M.c2, M.p2);
    M.p2 = 0.0f;
}

__device__ __forceinline__ void flush(HMember& M) {
    kahan_add(M.sx, M.cx_, M.px_);
    kahan_add(M.sy, M.cy_, M.py_);
    kahan_add(M.sz, M.cz_, M.pz_);
    kahan_add(M.su, M.cu, M.pu);
    M.px_ = M.py_ = M.pz_ = M.pu = 0.0f;
}

__device__ __forceinline__ void flush(VMember& M) {
    kahan_add(M.sd, M.cd, M.pd);
    kahan_add(M.sx, M.cx_, M.px_);
    kahan_add(M.sy, M.cy_, M.py_);
    kahan_add(M.sz, M.cz_, M.pz_);
    M.pd = M.px_ = M.py_ = M.pz_ = 0.0f;
}

__device__ __forceinline__ void flush(DVMember& M) {
    flush(static_cast<DMember&>(M));
    kahan_add(M.sd, M.cd, M.pd);
    kahan_add(M.sx, M.cx_, M.px_);
    kahan_add(M.sy, M.cy_, M.py_);
    kahan_add(M.sz, M.cz_, M.pz_);
    M.pd = M.px_ = M.py_ = M.pz_ = 0.0f;
}

__device__ __forceinline__ void flush(HAMember&) {}
__device__ __forceinline__ void flush(DAMember&) {}

template <class Mem>
__device__ __forceinline__ void precise_diff(const Mem& M, const SearchArgs& a, int crank, float& dx, float& dy,
                                             float& dz, float& r2) {
    uint4 Q = a.pfix[crank];
    float4 O = a.poff[crank];
    // the member's own fixed-point position, reloaded (rare path: no registers held)
    const uint4 P = a.pfix[M.rank];
    const float4 Om = a.poff[M.rank];
    dx = fix_diff(Q.x, O.x, P.x, Om.x);
    dy = fix_diff(Q.y, O.y, P.y, Om.y);
    dz = fix_diff(Q.z, O.z, P.z, Om.z);
    r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// density terms of a neighbour at q = r / h
__device__ __forceinline__ void density_terms(DMember& M, float mj, float q) {
    float w, v;
    m4_density(q, w, v);
    M.p0 = fmaf(mj, w, M.p0);
    M.p1 = fmaf(mj, v, M.p1);
}
__device__ __forceinline__ void density_terms(D2Member& M, float mj, float q) {
    float w, dw, d2w;
    m4_shape2(q, w, dw, d2w);
    M.p0 = fmaf(mj, w, M.p0);
    M.p1 = fmaf(mj, fmaf(q, dw, 3.0f * w), M.p1);
    M.p2 = fmaf(mj, fmaf(q * q, d2w, fmaf(8.0f * q, dw, 12.0f * w)), M.p2);
}

// Decision of the density criterion |r| < h_i, and the pair's difference.  The caller has
// counted the candidate in M.n; one that is outside is taken off and false returned.  Only
// the rare slow path branches: the FP64 re-test inside the band, and the exact
// differences of members far from the centre.
template <bool WRAP, class Mem>
__device__ __forceinline__ bool dens_decide(Mem& M, const SearchArgs& a, float3 p, int crank, LocalCounters& lc,
                                            float& dx, float& dy, float& dz, float& r2) {
    dx = rel_diff<WRAP>(p.x, M.mx);
    dy = rel_diff<WRAP>(p.y, M.my);
    dz = rel_diff<WRAP>(p.z, M.mz);
    r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    bool in = true;
    if (!(r2 < M.h2lo)) {
        in = false;
        if (r2 < M.h2hi) {
            const double e = exact_r2(a.xd, a.yd, a.zd, M.rank, crank);
            const double h = a.h64[M.rank];
            in = e < __dmul_rn(h, h);
            lc.retests++;
        }
        if (!in) M.n--;
        if (M.h2lo == kAlwaysSlow) precise_diff(M, a, crank, dx, dy, dz, r2);
    }
    return in;
}

// export of a pair: the next entry of the member's list
__device__ __forceinline__ void export_pair(MemberPos& M, const SearchArgs& a, int crank) {
    const int64_t q = M.xpos++;
    if (q < a.x_cap) a.x_idx[q] = a.perm[crank];
    else atomicOr(a.err, kErrCap);
}

// r from r^2 (1 ulp; 0 at 0)
__device__ __forceinline__ float sqrt_fast(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// density pair: p = candidate's coordinates relative to the member's centre, m_j its mass.
// A candidate outside enters the sums with mass 0 (phase A leaves few of them).
template <int MODE, bool WRAP = false, class Mem>
__device__ __forceinline__ void density_pair(Mem& M, const SearchArgs& a, float3 p, float mj, int crank,
                                             LocalCounters& lc) {
    float dx, dy, dz, r2;
    const bool in = dens_decide<WRAP>(M, a, p, crank, lc, dx, dy, dz, r2);
    if (MODE == kAcc) density_terms(M, in ? mj : 0.0f, q_of(sqrt_fast(r2), M.hinv));
    else if (MODE == kFill && in) export_pair(M, a, crank);
}

// divergence and curl terms of a neighbour at x_j - x_i = d: grad_i W = W'(r, h_i) (x_i -
// x_j) / r, v_ij = v_i - v_j; r^2 >= kMinR2 (grad W goes to 0 with r)
template <class Mem>
__device__ __forceinline__ void velocity_terms(Mem& M, float mj, float4 vj, float dx, float dy, float dz, float r2) {
    const float rinv = rsqrt_fast(r2);
    const float c = -M.sk * m4_slope(q_of(r2 * rinv, M.hinv)) * rinv;   // x_i - x_j = -d
    const float gx = c * dx, gy = c * dy, gz = c * dz;
    const float vx = M.vx - vj.x, vy = M.vy - vj.y, vz = M.vz - vj.z;
    M.pd = fmaf(-mj, fmaf(vx, gx, fmaf(vy, gy, vz * gz)), M.pd);
    M.px_ = fmaf(mj, fmaf(vy, gz, -vz * gy), M.px_);
    M.py_ = fmaf(mj, fmaf(vz, gx, -vx * gz), M.py_);
    M.pz_ = fmaf(mj, fmaf(vx, gy, -vy * gx), M.pz_);
}

// density pair with the velocity derivatives over the same decision
template <int MODE, bool WRAP = false>
__device__ __forceinline__ void densvel_pair(DVMember& M, const SearchArgs& a, float3 p, float mj, float4 vj,
                                             int crank, LocalCounters& lc) {
    float dx, dy, dz, r2;
    const bool in = dens_decide<WRAP>(M, a, p, crank, lc, dx, dy, dz, r2);
    if (MODE != kAcc) return;
    density_terms(M, in ? mj : 0.0f, q_of(sqrt_fast(r2), M.hinv));
    if (in && r2 >= kMinR2) velocity_terms(M, mj, vj, dx, dy, dz, r2);
}

// density pair of the recycled iteration: a candidate inside the widened threshold joins
// the member's sub-list, then the pair enters the sums at h as in density_pair
template <int MODE, bool WRAP = false>
__device__ __forceinline__ void density_list_pair(DLMember& M, const SearchArgs& a, float3 p, float mj, int crank,
                                                  LocalCounters& lc) {
    const float dx = rel_diff<WRAP>(p.x, M.mx), dy = rel_diff<WRAP>(p.y, M.my), dz = rel_diff<WRAP>(p.z, M.mz);
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    if (r2 < M.h2whi) {
        if (M.lcnt < M.lsub) M.lptr[M.lcnt] = crank;
        M.lcnt++;
    }
    density_pair<MODE, WRAP>(static_cast<DMember&>(M), a, p, mj, crank, lc);
}

// velocity-derivative pair (density criterion): p = relative coordinates, mj the mass,
// vj = {vx, vy, vz, -}
template <int MODE, bool WRAP = false>
__device__ __forceinline__ void vel_pair(VMember& M, const SearchArgs& a, float3 p, float mj, float4 vj, int crank,
                                         LocalCounters& lc) {
    float dx, dy, dz, r2;
    const bool in = dens_decide<WRAP>(M, a, p, crank, lc, dx, dy, dz, r2);
    if (MODE == kAcc && in && r2 >= kMinR2) velocity_terms(M, mj, vj, dx, dy, dz, r2);
}

// decision of the symmetric criterion |r| < max(h_i, h_j), as dens_decide
template <bool WRAP, class Mem>
__device__ __forceinline__ bool sym_decide(Mem& M, const SearchArgs& a, float3 p, float hj2, int crank,
                                           LocalCounters& lc, float& dx, float& dy, float& dz, float& r2) {
    dx = rel_diff<WRAP>(p.x, M.mx);
    dy = rel_diff<WRAP>(p.y, M.my);
    dz = rel_diff<WRAP>(p.z, M.mz);
    r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float H2 = fmaxf(M.h2, hj2);
    bool in = true;
    if (!(r2 < fmaf(H2, 1.0f - 3.0f * kBandRel, -M.bk))) {
        in = false;
        if (r2 < fmaf(H2, 1.0f + 3.0f * kBandRel, M.bk)) {
            const double e = exact_r2(a.xd, a.yd, a.zd, M.rank, crank);
            const double hi = a.h64[M.rank], hj = a.h64[crank];
            in = e < fmax(__dmul_rn(hi, hi), __dmul_rn(hj, hj));
            lc.retests++;
        }
        if (!in) M.n--;
        if (M.bk == -kAlwaysSlow) precise_diff(M, a, crank, dx, dy, dz, r2);
    }
    return in;
}

// hydro pair: p = relative coordinates, q = {h_j^2, m_j}, v = {vx, vy, vz, c_j},
// hh = {A_j, rho_j / 4, 1/h_j, limiter_j / 4}.  A pair below kMinR2 (coincident, or the member itself)
// has no kernel gradient.
template <int MODE, bool WRAP = false>
__device__ __forceinline__ void hydro_pair(HMember& M, const SearchArgs& a, float3 p, float2 q,
                                           float4 v, float4 hh, int crank, LocalCounters& lc) {
    // The member itself is a candidate, counted as a pair at r = 0 and taken off the
    // neighbour count at the end; the export skips it by rank.
    float dx, dy, dz, r2;
    const bool in = sym_decide<WRAP>(M, a, p, q.x, crank, lc, dx, dy, dz, r2);
    if (MODE == kFill && in && crank != M.rank) export_pair(M, a, crank);
    if (MODE != kAcc || !(in && r2 >= kMinR2)) return;
    const float rinv = rsqrt_fast(r2);
    const float r = r2 * rinv;
    const float dWi = M.sk * m4_slope(q_of(r, M.hinv));
    const float dWj = kSkernel * (hh.z * hh.z) * (hh.z * hh.z) * m4_slope(q_of(r, hh.z));
    const float rx = -dx, ry = -dy, rz = -dz;  // r_ij = x_i - x_j
    const float vx = M.vx - v.x, vy = M.vy - v.y, vz = M.vz - v.z;
    const float vr = fmaf(vx, rx, fmaf(vy, ry, vz * rz));
    // Pi = (-alpha cbar mu + beta mu^2) / rhobar for approaching pairs, rhobar = (rho_i +
    // rho_j) / 2, scaled by the pair mean of the limiter (1 for the plain viscosity).  The
    // records hold quarters of rho and the limiter, which cancel: the hardware reciprocal
    // flushes a subnormal result to zero, which 1 / (rho_i + rho_j) is above 2^126.
    const float hb = 0.5f * fmaf(q.x, hh.z, M.h);
    const float mu = hb * vr * rcp_fast(fmaf(a.eps * hb, hb, r2));
    const float cb = 0.5f * (M.cs + v.w);
    const float pi_ij = fmaf(-a.alpha * cb, mu, a.beta * mu * mu) * rcp_fast(M.rho4 + hh.y) * (M.fb4 + hh.w);
    const float visc = vr < 0.0f ? pi_ij : 0.0f;
    const float gbar = 0.5f * (dWi + dWj);
    const float mr = q.y * rinv;
    const float coef = mr * fmaf(M.A, dWi, fmaf(hh.x, dWj, visc * gbar));
    M.px_ = fmaf(coef, dx, M.px_);
    M.py_ = fmaf(coef, dy, M.py_);
    M.pz_ = fmaf(coef, dz, M.pz_);
    M.pu = fmaf(mr * fmaf(M.A, dWi, 0.5f * visc * gbar), vr, M.pu);
}

// Adjoint of sum_i w_i . a_i over one pair, gathered at member k.  The pair enters
// a_k and a_j through the symmetric factor B = A_k W'_k + A_j W'_j + Pi (W'_k + W'_j)/2
// (W' = dW/dr at h_k, h_j); their weighted sum is E = -B Q with
// Q = rhat . (m_j w_k - m_k w_j), rhat = (x_k - x_j) / r.  Accumulated: dE/d of x_k,
// v_k, m_k, h_k, rho_k (through the viscosity) and A_k.
template <int MODE, bool WRAP = false>
__device__ __forceinline__ void hydro_adj_pair(HAMember& M, const SearchArgs& a, float3 p, float2 q, float4 v,
                                               float4 hh, float4 wj, int crank, LocalCounters& lc) {
    // the member itself enters as a pair at r = 0, which contributes nothing
    float dx, dy, dz, r2;
    if (!sym_decide<WRAP>(M, a, p, q.x, crank, lc, dx, dy, dz, r2)) return;
    if (MODE != kAcc) return;
    if (r2 == 0.0f) return;
    const float rinv = rsqrt_any(r2);
    const float r = r2 * rinv;
    const float D0 = -dx, D1 = -dy, D2 = -dz;   // x_k - x_j
    const float e0 = D0 * rinv, e1 = D1 * rinv, e2 = D2 * rinv;
    float wk_, dwk, d2wk, wj_, dwj, d2wj;
    const float qk = q_of(r, M.hinv), qj = q_of(r, hh.z);
    m4_shape2(qk, wk_, dwk, d2wk);
    m4_shape2(qj, wj_, dwj, d2wj);
    const float Wr_k = M.sk * dwk, Wr_j = hh.w * dwj;
    const float Wrr_k = M.sk * M.hinv * d2wk, Wrr_j = hh.w * hh.z * d2wj;
    const float Wrh_k = -M.sk * M.hinv * fmaf(qk, d2wk, 4.0f * dwk);
    const float v0 = M.vx - v.x, v1 = M.vy - v.y, v2 = M.vz - v.z;
    const float vr = fmaf(v0, D0, fmaf(v1, D1, v2 * D2));
    const float hbar = 0.5f * fmaf(q.x, hh.z, M.h);
    const float Dn = fmaf(a.eps * hbar, hbar, r2);
    const float iDn = rcp_fast(Dn);
    const float irbar = 0.5f * rcp_fast(M.rho4 + hh.y);   // 1 / rhobar, from quarters as in hydro_pair
    float Pi = 0.0f, Pmu = 0.0f;
    if (vr < 0.0f) {
        const float cbar = 0.5f * (M.cs + v.w);
        const float mu = hbar * vr * iDn;
        Pi = fmaf(-a.alpha * cbar, mu, a.beta * mu * mu) * irbar;
        Pmu = fmaf(2.0f * a.beta, mu, -a.alpha * cbar) * irbar;
    }
    const float sdw = Wr_k + Wr_j;
    const float B = fmaf(M.A, Wr_k, fmaf(hh.x, Wr_j, 0.5f * Pi * sdw));
    const float mj = q.y;
    const float U0 = mj * M.wx - M.m * wj.x, U1 = mj * M.wy - M.m * wj.y, U2 = mj * M.wz - M.m * wj.z;
    const float Q = fmaf(e0, U0, fmaf(e1, U1, e2 * U2));
    M.mb = fmaf(B, fmaf(e0, wj.x, fmaf(e1, wj.y, e2 * wj.z)), M.mb);
    M.Ab = fmaf(-Q, Wr_k, M.Ab);
    float dmu_dh = 0.0f;
    if (vr < 0.0f) dmu_dh = 0.5f * vr * fmaf(-a.eps * hbar, hbar, r2) * iDn * iDn;
    M.hb = fmaf(-Q, fmaf(M.A, Wrh_k, fmaf(0.5f * Pi, Wrh_k, 0.5f * sdw * Pmu * dmu_dh)), M.hb);
    M.rb = fmaf(Q * Pi, 0.25f * sdw * irbar, M.rb);
    const float cm = 0.5f * sdw * Pmu;
    if (vr < 0.0f) {
        const float cv = -Q * cm * hbar * iDn;
        M.vb[0] = fmaf(cv, D0, M.vb[0]);
        M.vb[1] = fmaf(cv, D1, M.vb[1]);
        M.vb[2] = fmaf(cv, D2, M.vb[2]);
    }
    const float dBr = fmaf(M.A, Wrr_k, fmaf(hh.x, Wrr_j, 0.5f * Pi * (Wrr_k + Wrr_j)));
    const float ca = (vr < 0.0f) ? hbar * iDn : 0.0f;
    const float cb2 = (vr < 0.0f) ? -2.0f * hbar * vr * iDn * iDn : 0.0f;
    {
        const float dB = fmaf(dBr, e0, cm * fmaf(ca, v0, cb2 * D0));
        const float dQ = (U0 - Q * e0) * rinv;
        M.xb[0] = fmaf(-Q, dB, fmaf(-B, dQ, M.xb[0]));
    }
    {
        const float dB = fmaf(dBr, e1, cm * fmaf(ca, v1, cb2 * D1));
        const float dQ = (U1 - Q * e1) * rinv;
        M.xb[1] = fmaf(-Q, dB, fmaf(-B, dQ, M.xb[1]));
    }
    {
        const float dB = fmaf(dBr, e2, cm * fmaf(ca, v2, cb2 * D2));
        const float dQ = (U2 - Q * e2) * rinv;
        M.xb[2] = fmaf(-Q, dB, fmaf(-B, dQ, M.xb[2]));
    }
}

// Adjoint of sum_i (alpha_i rho_i + beta_i dRho_i/dh_i) at fixed h, gathered at member k:
// rho_k's own sum (x_k moves every pair) and the sums of every j with k in N_j (x_k and
// m_k enter as a neighbour).  q = {h_j^2, m_j}, d = {alpha_j, beta_j, 1/h_j, s_j}.
template <int MODE, bool WRAP = false>
__device__ __forceinline__ void dens_adj_pair(DAMember& M, const SearchArgs& a, float3 p, float2 q, float4 d,
                                              int crank, LocalCounters& lc) {
    // The member itself enters as a pair at r = 0 like any coincident neighbour:
    // alpha W(0, h) + beta W_h(0, h) = alpha s h - 3 beta s, and no position term.
    float dx, dy, dz, r2;
    if (!sym_decide<WRAP>(M, a, p, q.x, crank, lc, dx, dy, dz, r2)) return;
    if (MODE != kAcc) return;
    const float rinv = r2 >= kMinR2 ? rsqrt_fast(r2) : 0.0f;
    const float r = r2 * rinv;
    float wk_, dwk, d2wk, wj_, dwj, d2wj;
    const float qk = q_of(r, M.hinv), qj = q_of(r, d.z);
    m4_shape2(qk, wk_, dwk, d2wk);
    m4_shape2(qj, wj_, dwj, d2wj);
    // k as a neighbour of j: rho_j gains m_k W(r, h_j), dRho_j/dh_j gains m_k W_h(r, h_j)
    const float hj = q.x * d.z;
    M.mb = fmaf(d.x * d.w, hj * wj_, fmaf(-d.y * d.w, fmaf(qj, dwj, 3.0f * wj_), M.mb));
    if (r2 < kMinR2) return;
    const float Wr_k = M.sk * dwk, Wr_j = d.w * dwj;
    const float Whr_k = -M.sk * M.hinv * fmaf(qk, d2wk, 4.0f * dwk);
    const float Whr_j = -d.w * d.z * fmaf(qj, d2wj, 4.0f * dwj);
    const float coef = fmaf(M.alpha * q.y, Wr_k, fmaf(M.beta * q.y, Whr_k, fmaf(d.x * M.m, Wr_j, d.y * M.m * Whr_j)));
    const float c = -coef * rinv;   // rhat = (x_k - x_j) / r = -d / r
    M.xb[0] = fmaf(c, dx, M.xb[0]);
    M.xb[1] = fmaf(c, dy, M.xb[1]);
    M.xb[2] = fmaf(c, dz, M.xb[2]);
}

// phase B dispatch
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(DMember& M, const SearchArgs& a, const PlainTile& T, int j,
                                          LocalCounters& lc) {
    density_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), T.m[j], T.r[j], lc);
}
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(D2Member& M, const SearchArgs& a, const PlainTile& T, int j,
                                          LocalCounters& lc) {
    density_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), T.m[j], T.r[j], lc);
}
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(DVMember& M, const SearchArgs& a, const VelTile& T, int j,
                                          LocalCounters& lc) {
    densvel_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), T.m[j], T.v[j], T.r[j], lc);
}
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(DLMember& M, const SearchArgs& a, const PlainTile& T, int j,
                                          LocalCounters& lc) {
    density_list_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), T.m[j], T.r[j], lc);
}
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(VMember& M, const SearchArgs& a, const VelTile& T, int j,
                                          LocalCounters& lc) {
    vel_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), T.m[j], T.v[j], T.r[j], lc);
}
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(HMember& M, const SearchArgs& a, const HydroTile& T, int j,
                                          LocalCounters& lc) {
    hydro_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), make_float2(T.h2[j], T.m[j]), T.v[j], T.h[j], T.r[j], lc);
}
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(HAMember& M, const SearchArgs& a, const HAdjTile& T, int j,
                                          LocalCounters& lc) {
    hydro_adj_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), make_float2(T.h2[j], T.m[j]), T.v[j], T.h[j], T.wt[j], T.r[j], lc);
}
template <int MODE, bool WRAP>
__device__ __forceinline__ void tile_pair(DAMember& M, const SearchArgs& a, const DAdjTile& T, int j,
                                          LocalCounters& lc) {
    dens_adj_pair<MODE, WRAP>(M, a, make_float3(T.x[j], T.y[j], T.z[j]), make_float2(T.h2[j], T.m[j]), T.d[j], T.r[j], lc);
}

// Phase-A thresholds: of the dot form |p|^2 - 2 p.m (one-sided kinds: a constant of the
// member; symmetric ones: max(h^2, h_j^2) (1 + band) + bk_dot) and of the difference form
__device__ __forceinline__ float thr_dot(const DMember& M) { return M.thr_dot; }
__device__ __forceinline__ float thr_dot(const DLMember& M) { return M.thr_dot_w; }
__device__ __forceinline__ float thr_dot(const VMember& M) { return M.thr_dot; }
__device__ __forceinline__ float thr_dot(const SymMember& M) { return M.bk_dot; }
__device__ __forceinline__ float thr_diff(const DMember& M, float) { return M.h2hi; }
__device__ __forceinline__ float thr_diff(const DLMember& M, float) { return M.h2whi; }
__device__ __forceinline__ float thr_diff(const VMember& M, float) { return M.h2hi; }
__device__ __forceinline__ float thr_diff(const SymMember& M, float hj2) {
    return fmaf(fmaxf(M.h2, hj2), 1.0f + 3.0f * kBandRel, M.bk);   // precise members: everything
}

// combine the slice copies of a member: add the values held o lanes above, where add says so
struct SliceStep {
    int o;
    bool add;
};
__device__ __forceinline__ float xsum(float v, SliceStep o) {
    const float t = __shfl_down_sync(0xffffffffu, v, o.o);
    return o.add ? v + t : v;
}
__device__ __forceinline__ int xsum(int v, SliceStep o) {
    const int t = __shfl_down_sync(0xffffffffu, v, o.o);
    return o.add ? v + t : v;
}
__device__ __forceinline__ void slice_add(DMember& M, SliceStep o) {
    M.s0 = xsum(M.s0, o); M.c0 = xsum(M.c0, o); M.s1 = xsum(M.s1, o); M.c1 = xsum(M.c1, o);
    M.n = xsum(M.n, o);
}
__device__ __forceinline__ void slice_add(D2Member& M, SliceStep o) {
    slice_add(static_cast<DMember&>(M), o);
    M.s2 = xsum(M.s2, o); M.c2 = xsum(M.c2, o);
}
__device__ __forceinline__ void slice_add(DVMember& M, SliceStep o) {
    slice_add(static_cast<DMember&>(M), o);
    M.sd = xsum(M.sd, o); M.cd = xsum(M.cd, o); M.sx = xsum(M.sx, o); M.cx_ = xsum(M.cx_, o);
    M.sy = xsum(M.sy, o); M.cy_ = xsum(M.cy_, o); M.sz = xsum(M.sz, o); M.cz_ = xsum(M.cz_, o);
}
__device__ __forceinline__ void slice_add(HMember& M, SliceStep o) {
    M.sx = xsum(M.sx, o); M.cx_ = xsum(M.cx_, o); M.sy = xsum(M.sy, o); M.cy_ = xsum(M.cy_, o);
    M.sz = xsum(M.sz, o); M.cz_ = xsum(M.cz_, o); M.su = xsum(M.su, o); M.cu = xsum(M.cu, o);
    M.n = xsum(M.n, o);
}
__device__ __forceinline__ void slice_add(VMember& M, SliceStep o) {
    M.sd = xsum(M.sd, o); M.cd = xsum(M.cd, o); M.sx = xsum(M.sx, o); M.cx_ = xsum(M.cx_, o);
    M.sy = xsum(M.sy, o); M.cy_ = xsum(M.cy_, o); M.sz = xsum(M.sz, o); M.cz_ = xsum(M.cz_, o);
    M.n = xsum(M.n, o);
}
__device__ __forceinline__ void slice_add(HAMember& M, SliceStep o) {
    for (int k = 0; k < 3; ++k) { M.xb[k] = xsum(M.xb[k], o); M.vb[k] = xsum(M.vb[k], o); }
    M.mb = xsum(M.mb, o); M.hb = xsum(M.hb, o); M.rb = xsum(M.rb, o); M.Ab = xsum(M.Ab, o);
    M.n = xsum(M.n, o);
}
__device__ __forceinline__ void slice_add(DAMember& M, SliceStep o) {
    for (int k = 0; k < 3; ++k) M.xb[k] = xsum(M.xb[k], o);
    M.mb = xsum(M.mb, o);
    M.n = xsum(M.n, o);
}

// results of a member
template <int MODE>
__device__ __forceinline__ void write_result(const DMember& D, const SearchArgs& a) {
    if (MODE == kAcc) {
        a.o_s0[D.rank] = D.s0 - D.c0;
        a.o_s1[D.rank] = D.s1 - D.c1;
        a.o_n[D.rank] = D.n;
    } else if (MODE == kCount) {
        a.x_cnt[a.perm[D.rank]] = D.n;
    }
}
template <int MODE>
__device__ __forceinline__ void write_result(const D2Member& D, const SearchArgs& a) {
    write_result<MODE>(static_cast<const DMember&>(D), a);
    if (MODE == kAcc) a.o_s2[D.rank] = D.s2 - D.c2;
}
template <int MODE>
__device__ __forceinline__ void write_result(const DVMember& D, const SearchArgs& a) {
    write_result<MODE>(static_cast<const DMember&>(D), a);
    if (MODE == kAcc)
        a.o_vsum[D.rank] = make_float4(D.sd - D.cd, D.sx - D.cx_, D.sy - D.cy_, D.sz - D.cz_);
}
template <int MODE>
__device__ __forceinline__ void write_result(const HMember& H, const SearchArgs& a) {
    if (MODE == kAcc && a.o_res4) {
        // key order: the members of a group are consecutive ranks, so these writes are
        // contiguous; a gather pass moves them to the caller's order
        a.o_res4[H.rank] = make_float4(H.sx - H.cx_, H.sy - H.cy_, H.sz - H.cz_, H.su - H.cu);
        a.o_rcnt[H.rank] = H.n - 1;   // the member itself was counted as a pair
        return;
    }
    int orig = a.perm[H.rank];
    if (MODE == kAcc) {
        a.o_acc[3 * (int64_t)orig] = H.sx - H.cx_;
        a.o_acc[3 * (int64_t)orig + 1] = H.sy - H.cy_;
        a.o_acc[3 * (int64_t)orig + 2] = H.sz - H.cz_;
        a.o_dudt[orig] = H.su - H.cu;
        if (a.o_nh) a.o_nh[orig] = H.n - 1;   // the member itself was counted as a pair
    } else if (MODE == kCount) {
        a.x_cnt[orig] = H.n - 1;
    }
}
template <int MODE>
__device__ __forceinline__ void write_result(const HAMember& H, const SearchArgs& a) {
    if (MODE != kAcc) return;
    a.o_adj0[H.rank] = make_float4(H.xb[0], H.xb[1], H.xb[2], H.mb);
    a.o_adj1[H.rank] = make_float4(H.vb[0], H.vb[1], H.vb[2], 0.0f);
    a.o_adj2[H.rank] = make_float4(H.hb, H.rb, H.Ab, (float)H.n);
}
template <int MODE>
__device__ __forceinline__ void write_result(const VMember& V, const SearchArgs& a) {
    if (MODE != kAcc) return;
    a.o_res4[V.rank] = make_float4(V.rrho * (V.sd - V.cd), V.rrho * (V.sx - V.cx_), V.rrho * (V.sy - V.cy_),
                                   V.rrho * (V.sz - V.cz_));
}
template <int MODE>
__device__ __forceinline__ void write_result(const DAMember& D, const SearchArgs& a) {
    if (MODE != kAcc) return;
    a.o_adj3[D.rank] = make_float4(D.xb[0], D.xb[1], D.xb[2], D.mb);
}

// ---------------------------------------------------------------------------------
// Grouped form: one warp per group
// ---------------------------------------------------------------------------------

struct alignas(16) WalkSmem {
    uint32_t stack[kStackCap];   // node ranges: (first child << 3) | (count - 1)
    int2 ranges[kRangeCap];      // ring of pending particle ranges {first rank - flat start, flat start}
    WalkCounters ctr;            // written by lane 0
};

__device__ __forceinline__ void clear_counters(WalkSmem& W, int lane) {
    if (lane == 0) W.ctr = WalkCounters{0u, 0u, 0u, 0u};
}

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Member slot layout of a lane: the part's gw members in S copies ("slices"), each
// filtering a different subset of the candidates; k = the lane's member, -1 if it holds
// none (its slice is then S or more, or the member has left).
struct Layout {
    int gw, S, slice, k;
    int rows;       // quads of candidates a slice holds
    uint32_t inv;   // ceil(2^16 / S): n / S = n * inv >> 16 for the n <= 2^10 used here
};

// pow2: member slots rounded up to a power of two and at most 4 slices
__device__ __forceinline__ Layout make_layout(int cnt, int lane, bool allow_slices, int max_slices, bool pow2,
                                              int tile) {
    Layout L;
    L.gw = pow2 && cnt > 1 ? 1 << (32 - __clz(cnt - 1)) : cnt;
    const uint32_t q = 65536u / (uint32_t)L.gw + 1u;
    L.S = allow_slices ? min((int)((32u * q) >> 16), max_slices) : 1;
    L.slice = (int)(((uint32_t)lane * q) >> 16);
    const int k = lane - L.slice * L.gw;
    L.k = (L.slice < L.S && k < cnt) ? k : -1;
    L.inv = 65535u / (uint32_t)L.S + 1u;
    L.rows = (int)(((tile / 4) * L.inv) >> 16);
    return L;
}

// sum over the slices, ending in slice 0: halves folded onto each other
template <class Mem>
__device__ __forceinline__ void slice_sum(Mem& M, const Layout& L) {
    for (int n = L.S; n > 1;) {
        const int half = (n + 1) >> 1;
        slice_add(M, SliceStep{half * L.gw, L.slice + half < n});
        n = half;
    }
}

// place of the t-th candidate of a tile
__device__ __forceinline__ int tile_place(const Layout& L, int t) {
    const int quad = t >> 2;
    const int row = (int)((quad * L.inv) >> 16);
    return ((quad - row * L.S) * L.rows + row) * 4 + (t & 3);
}

// Phase A of one mask word: 4 * quads of the lane's candidates from place j0 against the
// member's FP32 threshold, the first in the top bit of the 4 * quads lowest ones (quads
// even).  Dot form, packed: per quad four 16-byte shared-memory loads, six packed FMAs, two
// packed adds and four shifts that collect the signs; its rounding stays inside the FP64
// decision band.
template <class K, bool WRAP>
__device__ __forceinline__ uint32_t test_word(const typename K::Tile& T, const typename K::Member& Mb, int j0,
                                              int quads) {
    uint32_t mask = 0u;
    if constexpr (!WRAP) {
        const unsigned long long ax = pair_of(-2.0f * Mb.mx, -2.0f * Mb.mx), ay = pair_of(-2.0f * Mb.my, -2.0f * Mb.my),
                                 az = pair_of(-2.0f * Mb.mz, -2.0f * Mb.mz),
                                 at = pair_of(-thr_dot(Mb), -thr_dot(Mb));
        for (int r = 0; r < quads; r += 2) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int j = j0 + 4 * (r + q);
                const ulonglong2 px = *reinterpret_cast<const ulonglong2*>(&T.x[j]);
                const ulonglong2 py = *reinterpret_cast<const ulonglong2*>(&T.y[j]);
                const ulonglong2 pz = *reinterpret_cast<const ulonglong2*>(&T.z[j]);
                const ulonglong2 pw = *reinterpret_cast<const ulonglong2*>(&T.w[j]);
                unsigned long long t0 = add_pair(pw.x, at), t1 = add_pair(pw.y, at);
                if constexpr (K::sym) {
                    const float4 hj2 = *reinterpret_cast<const float4*>(&T.h2[j]);
                    constexpr float kk = -(1.0f + 3.0f * kBandRel);
                    t0 = fma_pair(pair_of(fmaxf(Mb.h2, hj2.x), fmaxf(Mb.h2, hj2.y)), pair_of(kk, kk), t0);
                    t1 = fma_pair(pair_of(fmaxf(Mb.h2, hj2.z), fmaxf(Mb.h2, hj2.w)), pair_of(kk, kk), t1);
                }
                t0 = fma_pair(px.x, ax, fma_pair(py.x, ay, fma_pair(pz.x, az, t0)));
                t1 = fma_pair(px.y, ax, fma_pair(py.y, ay, fma_pair(pz.y, az, t1)));
                mask = push_sign(mask, (uint32_t)t0);
                mask = push_sign(mask, (uint32_t)(t0 >> 32));
                mask = push_sign(mask, (uint32_t)t1);
                mask = push_sign(mask, (uint32_t)(t1 >> 32));
            }
        }
    } else {
        for (int j = j0; j < j0 + 4 * quads; ++j) {
            float hj2 = 0.0f;
            if constexpr (K::sym) hj2 = T.h2[j];
            const float dx = rel_diff<true>(T.x[j], Mb.mx), dy = rel_diff<true>(T.y[j], Mb.my),
                        dz = rel_diff<true>(T.z[j], Mb.mz);
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            mask = (mask << 1) | (r2 < thr_diff(Mb, hj2) ? 1u : 0u);
        }
    }
    return mask;
}

// Member x candidate filter of the nt candidates in the tile.  Phase A: bit masks of the
// lane's slice, a word per 32 candidates; their bits count as neighbours.  Phase B: every
// lane walks its own set bits across all words (no per-word wait for the slowest lane)
// for the exact decision and the pair terms; forward partial sums are folded into the
// compensated totals after the tile.
template <class K, int MODE, bool WRAP>
__device__ __forceinline__ void filter_tile(typename K::Tile& T, const Layout& L, typename K::Member& Mb, int nt,
                                            const SearchArgs& a, LocalCounters& lc, int lane) {
    const int S = L.S;
    const int full = nt >> 2;                                             // whole quads
    const int most = (int)((((nt + 3) >> 2) + S - 1) * L.inv >> 16);      // quads of slice 0, the longest
    // the lane's own candidates: its whole quads, and the last part quad if it is its
    int mine = 0;
    if (Mb.rank >= 0) {
        const int own = (int)((full + S - 1 - L.slice) * L.inv >> 16);
        const bool part = (int)((full + S - L.slice) * L.inv >> 16) != own;
        mine = 4 * own + (part ? nt & 3 : 0);
    }
    lc.tests += mine;
    const int nw = (most + 7) >> 3;
    // lanes without a member test slice 0's and drop it
    const int j0 = (L.slice < S ? L.slice : 0) * L.rows * 4;
    int hits = 0;
    for (int c = 0; c < nw; ++c) {
        const int quads = min(8, (most - 8 * c + 1) & ~1);
        const int own = min(max(mine - 32 * c, 0), 32);
        const uint32_t mask = (test_word<K, WRAP>(T, Mb, j0 + 32 * c, quads) << (32 - 4 * quads)) &
                              (uint32_t)(0xffffffff00000000ull >> own);
        T.masks[(c << 5) + lane] = mask;
        hits += __popc(mask);
    }
    Mb.n += hits;
    // two words at a time in registers, the second following the first without a branch
    for (int c = 0; c < nw; c += 2) {
        uint32_t cur = T.masks[(c << 5) + lane], nxt = c + 1 < nw ? T.masks[(c << 5) + 32 + lane] : 0u;
        int j1 = j0 + (c << 5);
        while (cur | nxt) {
            if (cur == 0u) {
                cur = nxt;
                nxt = 0u;
                j1 += 32;
            }
            const int q = __clz(cur);
            cur &= 0x7fffffffu >> q;
            tile_pair<MODE, WRAP>(Mb, a, T, j1 + q, lc);
        }
    }
    if (MODE == kAcc) flush(Mb);
}

// Work item of the grouped kernels: members U[base, base + cnt), or the set bits of `mask`
// as offsets from base (pieces of at most 32 entries; mask 0: the range), the walk's
// start node (a root of the forest) and the slice limit.
struct GroupDesc {
    int base, cnt;
    uint32_t mask;
    int root, smax;
};

// entry of the piece list for item gid: the large pieces, listed from the end, go first
__device__ __forceinline__ int64_t piece_index(const SearchArgs& a, int gid, int nlarge) {
    return gid < nlarge ? a.pieces_cap - 1 - gid : gid - nlarge;
}

__device__ __forceinline__ GroupDesc group_desc(const SearchArgs& a, int gid, int nlarge) {
    GroupDesc d;
    d.root = 0;
    d.smax = 32;
    d.mask = 0u;
    if (a.pieces4) {
        const int4 G = a.pieces4[piece_index(a, gid, nlarge)];
        d.base = G.x;
        d.mask = (uint32_t)G.y;
        d.cnt = __popc(d.mask);
        d.root = G.z;
        const int s = (G.w >> 8) & 0xff;   // bits 16.. carry the box's leaf size
        d.smax = s >= 4 ? 32 : s;          // 4, the largest limit that can be set: all lanes
    } else if (a.pieces) {
        const int2 G = a.pieces[piece_index(a, gid, nlarge)];
        d.base = G.x;
        d.mask = (uint32_t)G.y;
        d.cnt = __popc(d.mask);
    } else {
        // a group of more than 32 members is `parts` items of 32
        const int k = a.parts > 1 ? gid / a.parts : gid;
        if (a.groups) {
            const int2 G = a.groups[k];
            d.base = G.x;
            d.cnt = G.y;
        } else {
            d.base = k * a.g;
            d.cnt = min(a.g, a.nu - d.base);
        }
        if (a.parts > 1) {
            const int b = (gid - k * a.parts) * kPartMax;
            d.base += b;
            d.cnt = min(d.cnt - b, kPartMax);
        }
    }
    return d;
}

// items of the launch, and how many of them are large pieces
__device__ __forceinline__ int group_count(const SearchArgs& a, int& nlarge) {
    nlarge = 0;
    if (!a.npieces) return a.ngroups * max(a.parts, 1);
    nlarge = a.npieces[1];
    return a.npieces[0] + nlarge;
}

// Group centre: the fixed-point position of the lowest lane that holds a member, or the
// centre of the members' bounding box (offsets from that member are exact minimum-image
// integers).  Every lane passes one record per slot; false when no lane holds a member.
template <int M>
__device__ __forceinline__ bool group_centre(const SearchArgs& a, const MemberRec (&rec)[M], uint32_t& cx,
                                             uint32_t& cy, uint32_t& cz) {
    const unsigned have = __ballot_sync(0xffffffffu, rec[0].rank >= 0);   // slot 0 holds the first members
    if (have == 0u) return false;
    const int ref = __ffs(have) - 1;
    cx = __shfl_sync(0xffffffffu, rec[0].P.x, ref);
    cy = __shfl_sync(0xffffffffu, rec[0].P.y, ref);
    cz = __shfl_sync(0xffffffffu, rec[0].P.z, ref);
    if (a.centre_box) {
        int lox = 0, loy = 0, loz = 0, hix = 0, hiy = 0, hiz = 0;
#pragma unroll
        for (int mm = 0; mm < M; ++mm) {
            if (rec[mm].rank >= 0) {
                const int dx = (int32_t)(rec[mm].P.x - cx), dy = (int32_t)(rec[mm].P.y - cy),
                          dz = (int32_t)(rec[mm].P.z - cz);
                lox = min(lox, dx); hix = max(hix, dx);
                loy = min(loy, dy); hiy = max(hiy, dy);
                loz = min(loz, dz); hiz = max(hiz, dz);
            }
        }
        lox = __reduce_min_sync(0xffffffffu, lox);
        loy = __reduce_min_sync(0xffffffffu, loy);
        loz = __reduce_min_sync(0xffffffffu, loz);
        hix = __reduce_max_sync(0xffffffffu, hix);
        hiy = __reduce_max_sync(0xffffffffu, hiy);
        hiz = __reduce_max_sync(0xffffffffu, hiz);
        cx += (uint32_t)(int32_t)(((int64_t)lox + hix) >> 1);
        cy += (uint32_t)(int32_t)(((int64_t)loy + hiy) >> 1);
        cz += (uint32_t)(int32_t)(((int64_t)loz + hiz) >> 1);
    }
    return true;
}

// 6-bit v spread so that bit b lands on bit 3b
__device__ __forceinline__ uint32_t spread6(uint32_t v) {
    v = (v | (v << 8)) & 0x300fu;
    v = (v | (v << 4)) & 0x30c3u;
    return (v | (v << 2)) & 0x9249u;
}

// First nodes of the walk, one per lane (-1: none): the nodes of the up to eight cells of
// one octree level (<= kStartLevels) that the cube of half width Rb (box units) around C,
// which covers the whole search region, can meet (tab: the start table of the tree rooted
// at `root`).  The level is the deepest whose cells are at least as wide as the cube, so
// it meets at most two per axis; every particle within the region lies in one of
// those cells and hence in its node's subtree.  A cell without a node of its own is
// empty, unless an ancestor is a leaf: then that leaf, once.
__device__ __forceinline__ int walk_start(const SearchArgs& a, int root, uint32_t cx, uint32_t cy, uint32_t cz,
                                          float Rb, int lane) {
    static_assert(kStartLevels <= 6, "spread6 takes 6 bits per axis");
    // half width in fixed-point units, rounded up, plus the sub-unit offsets of the positions
    const float Ru = __fmul_ru(__fmul_ru(Rb, 1.000002f), 4294967296.0f);
    int node = lane == 0 ? root : -1;
    if (!a.start_tab || !(Ru < 1.07e9f)) return node;   // below a quarter of the box (2^30): level >= 1
    const uint32_t r = (uint32_t)Ru + 3u;
    int lvl = min(kStartLevels, __clz(2u * r));
    const int sh = 32 - lvl;
    const uint32_t x0 = (cx - r) >> sh, y0 = (cy - r) >> sh, z0 = (cz - r) >> sh;
    const uint32_t x1 = (cx + r) >> sh, y1 = (cy + r) >> sh, z1 = (cz + r) >> sh;
    const bool bx = lane & 4, by = lane & 2, bz = lane & 1;
    node = -1;
    if (lane < 8 && !(bx && x0 == x1) && !(by && y0 == y1) && !(bz && z0 == z1)) {
        const int32_t* tab = a.start_tab + (size_t)root * kStartTableSize;
        uint32_t m = (spread6(bx ? x1 : x0) << 2) | (spread6(by ? y1 : y0) << 1) | spread6(bz ? z1 : z0);
        node = tab[start_table_offset(lvl) + m];
        const bool own = node >= 0;
        while (node < 0) {
            m >>= 3;
            --lvl;
            node = lvl >= 1 ? tab[start_table_offset(lvl) + m] : root;
        }
        if (!own && a.nlink[node].z >= 0) node = -1;
    }
    const unsigned same = __match_any_sync(0xffffffffu, node);
    return (node >= 0 && lane == __ffs(same) - 1) ? node : -1;
}

// The walk's stack and the ring of particle ranges it emits.  The stack lives in shared
// memory (at most a.stack_cap entries); when it fills up, its oldest entries move to this
// warp's overflow area in global memory, which holds the bottom of the stack and refills
// the shared part when that runs empty.  The ranges, laid end to end in walk order, number
// the candidates flat: [done, total) are pending, in ring entries [e0, e1).
struct Walk {
    int sp, gsp;
    int e0, e1, done, total;

    __device__ __forceinline__ bool empty() const { return sp == 0 && gsp == 0; }
};

__device__ __forceinline__ uint32_t* walk_overflow(const SearchArgs& a) {
    return a.stack_spill + (size_t)(blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5)) * kSpillCap;
}

__device__ __forceinline__ Walk walk_begin() {
    Walk w;
    w.sp = w.gsp = 0;
    w.e0 = w.e1 = w.done = w.total = 0;
    return w;
}

// A step can be taken: entries on the stack, room to push 32 of them and to emit 32 ranges.
__device__ __forceinline__ bool walk_can_step(const SearchArgs& a, const Walk& w) {
    return !w.empty() && w.sp <= a.stack_cap - 32 && w.e1 - w.e0 <= kRangeCap - 32;
}

// One node per lane (-1: none) is tested (open_node(have, cen, ext, candidates so far),
// called by all lanes); of the open ones, leaves and nodes of at most `whole` particles emit
// their range, the others push their children.
template <class Open>
__device__ __forceinline__ void walk_visit(const SearchArgs& a, WalkSmem& W, Walk& w, int node, int whole,
                                           int lane, Open open_node) {
    const uint32_t lt = (1u << lane) - 1u;
    bool emit = false, push = false;
    int4 lk = make_int4(0, 0, -1, 0);
    int nch = 0;
    uint4 cen = make_uint4(0u, 0u, 0u, 0u);
    float4 ext = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (node >= 0) {
        cen = a.ncen[node];
        ext = a.next[node];
        lk = a.nlink[node];
        nch = __float_as_int(ext.w);
    }
    const bool open = open_node(node >= 0, cen, ext, w.total);
    emit = open && lk.y > 0 && (lk.z < 0 || lk.y <= whole);
    push = open && lk.z >= 0 && !emit;
    const int nn = __popc(__ballot_sync(0xffffffffu, node >= 0));
    if (lane == 0) W.ctr.nodes += nn;
    const unsigned em = __ballot_sync(0xffffffffu, emit);
    if (em) {
        const int add = emit ? lk.y : 0;
        const int pre = warp_incl_scan(add, lane);
        if (emit) {
            const int start = w.total + pre - add;
            W.ranges[(w.e1 + __popc(em & lt)) & (kRangeCap - 1)] = make_int2(lk.x - start, start);
        }
        w.e1 += __popc(em);
        w.total += __shfl_sync(0xffffffffu, pre, 31);
    }
    const unsigned pm = __ballot_sync(0xffffffffu, push);
    if (push) W.stack[w.sp + __popc(pm & lt)] = ((uint32_t)lk.z << 3) | (uint32_t)(nch - 1);
    w.sp += __popc(pm);
    if (lane == 0) W.ctr.deep = max(W.ctr.deep, (unsigned)(w.sp + w.gsp));
    __syncwarp();
}

// One step: the children of up to four entries from the top of the stack, eight lanes to
// an entry.
template <class Open>
__device__ __forceinline__ void walk_step(const SearchArgs& a, WalkSmem& W, Walk& w, int whole, int lane,
                                          Open open_node) {
    if (w.sp == 0) {
        const int m = min(w.gsp, 32);
        if (lane < m) W.stack[lane] = walk_overflow(a)[w.gsp - m + lane];
        w.gsp -= m;
        w.sp = m;
        __syncwarp();
    }
    const int e = w.sp - 1 - (lane >> 3);
    int node = -1;
    if (e >= 0) {
        const uint32_t ent = W.stack[e];
        if ((uint32_t)(lane & 7) <= (ent & 7u)) node = (int)(ent >> 3) + (lane & 7);
    }
    w.sp = max(w.sp - 4, 0);
    __syncwarp();
    walk_visit(a, W, w, node, whole, lane, open_node);
}

// When the next step could push more entries than the shared part holds, the oldest (up
// to 32, its bottom) move to the top of the overflow area, which stays below the shared
// part, so the whole stack remains last in, first out.
__device__ __forceinline__ void walk_spill(const SearchArgs& a, WalkSmem& W, Walk& w, int lane) {
    if (w.sp <= a.stack_cap - 32) return;
    const int ev = min(32, w.sp);
    if (w.gsp + ev > kSpillCap) atomicOr(a.err, kErrStack);
    else if (lane < ev) walk_overflow(a)[w.gsp + lane] = W.stack[lane];
    __syncwarp();
    for (int b = 0; b < w.sp - ev; b += 32) {
        const uint32_t v = (b + lane < w.sp - ev) ? W.stack[ev + b + lane] : 0u;
        __syncwarp();
        if (b + lane < w.sp - ev) W.stack[b + lane] = v;
        __syncwarp();
    }
    w.gsp = min(w.gsp + ev, kSpillCap);
    w.sp -= ev;
}

// The next up to 32 pending candidates, one per lane: returns their number and this
// lane's rank (undefined beyond the number).  Lane l looks at range e0 + l; a window bit
// marks where each range starts, and a lane's range is the last one starting at or
// before it.  Only 32 ranges are looked at, so the window ends where the 33rd starts.
__device__ __forceinline__ int walk_take(WalkSmem& W, Walk& w, int lane, int& rank) {
    const int ne = w.e1 - w.e0;
    int take = min(32, w.total - w.done);
    if (ne > 32) take = min(take, W.ranges[(w.e0 + 32) & (kRangeCap - 1)].y - w.done);
    int2 R = make_int2(0, 0x7fffffff);
    if (lane < ne) R = W.ranges[(w.e0 + lane) & (kRangeCap - 1)];
    const int rel = lane < ne ? R.y - w.done : 64;
    const int first = __popc(__ballot_sync(0xffffffffu, rel <= 0)) - 1;   // the range holding candidate `done`
    const unsigned starts = __reduce_or_sync(0xffffffffu, (rel > 0 && rel < 32) ? 1u << rel : 0u);
    const int off = first + __popc(starts & ((2u << lane) - 1u));
    rank = __shfl_sync(0xffffffffu, R.x, off & 31) + w.done + lane;
    w.e0 += __popc(__ballot_sync(0xffffffffu, rel <= take)) - 1;
    w.done += take;
    __syncwarp();
    return take;
}

// A group beside a dense clump can have the clump within H of its box, and thousands of
// candidates, though no member's own sphere meets it.  Testing every node against every
// member costs about as much as the rest of a step per 8 members, so it starts when a walk
// has found kRefineBase + kRefinePerMember * members candidates (three times what an even
// density gives).  A density pass of 414k actives in runs among 2.1M clustered particles
// had groups of up to 10^4 candidates for 345 pairs, which ran for 0.4 ms of its 0.7 ms.
constexpr int kRefineBase = 256;
constexpr int kRefinePerMember = 48;

// Whether every lane's node (centre d relative to the group's, half extents in units, largest
// h) meets a member's sphere (lane k < gw: {m, radius}, radius 0: none).  Called by all
// lanes; not inlined, so that its registers are not held by the walk, which rarely comes
// here.  Margins of 1e-6 cover the FP32 errors of the coordinates.
__device__ __noinline__ bool meets_members(float3 d, float4 ext, float hnode, float4 mine, int gw) {
    const float slack = 1.0e-6f * (warp_max(fmaxf(fabsf(mine.x), fmaxf(fabsf(mine.y), fabsf(mine.z)))) + warp_max(mine.w));
    constexpr float kUp = 1.000001f * kUnitToBox;
    const float wx = fmaf(ext.x, kUp, slack), wy = fmaf(ext.y, kUp, slack), wz = fmaf(ext.z, kUp, slack);
    bool any = false;
    for (int k = 0; k < gw; ++k) {
        // nearest image of the node's centre, less the half extent
        const float ax = fabsf(d.x - __shfl_sync(0xffffffffu, mine.x, k)),
                    ay = fabsf(d.y - __shfl_sync(0xffffffffu, mine.y, k)),
                    az = fabsf(d.z - __shfl_sync(0xffffffffu, mine.z, k));
        const float gx = fmaxf(fminf(ax, 1.0f - ax) - wx, 0.0f), gy = fmaxf(fminf(ay, 1.0f - ay) - wy, 0.0f),
                    gz = fmaxf(fminf(az, 1.0f - az) - wz, 0.0f);
        float r = __shfl_sync(0xffffffffu, mine.w, k);
        r = r > 0.0f ? fmaxf(r, hnode) : 0.0f;
        any = any || fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < 1.000004f * r * r;
    }
    return any;
}

// One search's walk from the tree rooted at `root` and the member x candidate filter of
// every tile (the members are initialised relative to the centre C).
//
// A node or a candidate matters only if it lies within H of the members' box (H the
// largest member radius; symmetric kinds: or its own h), so both are tested against the
// box dilated by H.  The box is symmetric about C, E = max |m| per axis.  The sphere
// around C that covers every member's sphere is up to a third larger in volume for a
// cubic box and far larger for an elongated one.
//
// Bound by instruction issue (84% of the issue slots in the density loop, 74% in hydro; L2 hit
// 94%).  Of the about 900 particles
// that the opened nodes hold (16.8M clustered particles, g = 16) fewer than half lie in
// the dilated box: they are dropped here, at a few instructions per 32 of them, before
// the members' filter, and only the kept ones fetch the kind's own records.  Against
// staging every candidate of the covering sphere's leaves by bulk copies and filtering
// them all: a timestep of 16.8M clustered particles 128.8 -> 99.0 ms, hydro of 4.2M 10.9 -> 8.5 ms.
template <class K, int MODE>
__device__ __forceinline__ void group_search(const SearchArgs& a, WalkSmem& W, typename K::Tile& T, const Layout& L,
                                             typename K::Member& mem, uint32_t cx, uint32_t cy, uint32_t cz, int root,
                                             LocalCounters& lc, int lane) {
    const uint32_t lt = (1u << lane) - 1u;
    const float ex = warp_max(fabsf(mem.mx)), ey = warp_max(fabsf(mem.my)), ez = warp_max(fabsf(mem.mz));
    const float H = warp_max(member_radius(mem));
    // node test: half extents in fixed-point units, covering the FP32 error of the members'
    // coordinates (2 ulps and the rounding of the offset)
    const float nx = __fadd_ru(__fmul_ru(__fmul_ru(ex, 1.000001f), 4294967296.0f), 1.0f);
    const float ny = __fadd_ru(__fmul_ru(__fmul_ru(ey, 1.000001f), 4294967296.0f), 1.0f);
    const float nz = __fadd_ru(__fmul_ru(__fmul_ru(ez, 1.000001f), 4294967296.0f), 1.0f);
    const float H2u = radius2_units(H);
    // candidate test: the FP32 gap to the box is at most the FP32 distance to any member, so
    // the decision band of that distance covers it (|m| <= |E|)
    const float H2 = H * H;
    const float band = 8.0f * kBandRel * fmaf(ex, ex, fmaf(ey, ey, ez * ez));
    // every relevant pair difference is already the nearest image when the group's
    // reach stays below half the box (symmetric: with the largest h of the tree)
    const float emax = fmaxf(ex, fmaxf(ey, ez));
    const float reach = emax + (K::sym ? fmaxf(H, __uint_as_float(a.ncen[root].w)) : H);
    const bool wrap_safe = reach < 0.49f;
    auto open_box = [&](const uint4& cen, const float4& ext) {
        const float gap2 = node_gap2(cen, make_float4(__fadd_ru(ext.x, nx), __fadd_ru(ext.y, ny),
                                                      __fadd_ru(ext.z, nz), 0.0f), cx, cy, cz);
        if constexpr (K::sym) return gap2 <= radius2_units(fmaxf(H, __uint_as_float(cen.w)));
        else return gap2 <= H2u;
    };
    // candidates after which the walk also tests nodes against the members' own spheres
    const int refine_after = kRefineBase + kRefinePerMember * L.gw;
    auto open_node = [&](bool have, const uint4& cen, const float4& ext, int found) {
        bool open = have && open_box(cen, ext);
        if (found > refine_after)
            open = meets_members(make_float3(rel_coord(cen.x, 0.0f, cx), rel_coord(cen.y, 0.0f, cy),
                                             rel_coord(cen.z, 0.0f, cz)),
                                 ext, K::sym ? __uint_as_float(cen.w) : 0.0f,
                                 make_float4(mem.mx, mem.my, mem.mz, member_radius(mem)), L.gw) && open;
        return open;
    };
    const int whole = L.gw == 1 ? kWalkWholeSingle : kWalkWhole;
    Walk w = walk_begin();
    walk_visit(a, W, w, walk_start(a, root, cx, cy, cz, reach, lane), whole, lane, open_node);
    int ns = 0;                                 // candidates in the tile
    const int room = 4 * L.S * L.rows - 32;     // a window more still fits
    for (;;) {
        while (walk_can_step(a, w) && w.total - w.done < 64) walk_step(a, W, w, whole, lane, open_node);
        walk_spill(a, W, w, lane);
        const bool walked = w.empty();
        // candidates by whole windows of 32 while the walk goes on
        while (ns <= room && (w.total - w.done >= 32 || (walked && w.total > w.done))) {
            int rank;
            const int nt = walk_take(W, w, lane, rank);
            bool in = false;
            float px = 0.0f, py = 0.0f, pz = 0.0f, mj = 0.0f, hj2 = 0.0f;
            if (lane < nt) {
                const uint4 P = a.pfix[rank];
                const float4 O = a.poff[rank];
                px = rel_coord(P.x, O.x, cx);
                py = rel_coord(P.y, O.y, cy);
                pz = rel_coord(P.z, O.z, cz);
                mj = O.w;
                const float gx = fmaxf(fabsf(px) - ex, 0.0f), gy = fmaxf(fabsf(py) - ey, 0.0f),
                            gz = fmaxf(fabsf(pz) - ez, 0.0f);
                const float gap2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
                float lim = H2;
                if constexpr (K::sym) {
                    const float hj = __uint_as_float(P.w);
                    hj2 = hj * hj;
                    lim = fmaxf(H2, hj2);
                }
                in = gap2 < fmaf(lim, 1.0f + 3.0f * kBandRel, band);
            }
            const unsigned im = __ballot_sync(0xffffffffu, in);
            if (in) {
                const int t = tile_place(L, ns + __popc(im & lt));
                T.x[t] = px;
                T.y[t] = py;
                T.z[t] = pz;
                T.w[t] = fmaf(px, px, fmaf(py, py, pz * pz));
                T.m[t] = mj;
                if constexpr (K::sym) T.h2[t] = hj2;
                T.r[t] = rank;
                stage_records(T, a, t, rank);
            }
            ns += __popc(im);
        }
        const bool last = walked && w.total == w.done;
        if (last && lane == 0) W.ctr.cands += w.total;
        if (ns > room || last) {
            if (ns > 0) {
                copies_wait();
                __syncwarp();
                if (wrap_safe) filter_tile<K, MODE, false>(T, L, mem, ns, a, lc, lane);
                else filter_tile<K, MODE, true>(T, L, mem, ns, a, lc, lane);
                __syncwarp();
            }
            ns = 0;
            if (last) break;
        }
    }
}

// work-list entry of the lane's member
__device__ __forceinline__ int member_entry(const GroupDesc& d, const Layout& L, WalkSmem& W, int lane) {
    if (d.mask == 0u) return d.base + L.k;
    // member index -> offset, through the walk stack (free between searches)
    if (d.mask >> lane & 1u) W.stack[__popc(d.mask & ((1u << lane) - 1u))] = (uint32_t)lane;
    __syncwarp();
    const int off = (int)W.stack[max(L.k, 0)];
    __syncwarp();
    return d.base + off;
}

// The search of up to 32 members, one per lane and slice.
template <class K, int MODE>
__device__ __forceinline__ void process_part(const SearchArgs& a, WalkSmem& W, typename K::Tile& T, const GroupDesc& d,
                                             LocalCounters& lc, int lane) {
    constexpr bool kLists = K::id == kKindDensityList;
    const Layout L = make_layout(d.cnt, lane, MODE == kAcc, kLists ? min(4, d.smax) : d.smax, kLists,
                                 K::Tile::cap);
    const int entry = member_entry(d, L, W, lane);
    const MemberRec rec[1] = {load_member(a, L.k >= 0 ? a.U[entry] : -1)};
    uint32_t cx = 0, cy = 0, cz = 0;
    if (!group_centre<1>(a, rec, cx, cy, cz)) return;
    typename K::Member mem;
    member_init(mem, a, rec[0], cx, cy, cz);
    if constexpr (kLists) {
        // list slot = the member's index in the work list; sub-list of this lane's slice
        if (mem.rank >= 0) {
            mem.lsub = kListCap / L.S;
            mem.lptr = a.o_list + (int64_t)entry * kListCap + L.slice * mem.lsub;
        }
    }
    // export: write position of the member's neighbours
    if (MODE == kFill && mem.rank >= 0) mem.xpos = a.x_off[a.perm[mem.rank]];
    if (lane == 0) W.ctr.walks++;
    group_search<K, MODE>(a, W, T, L, mem, cx, cy, cz, d.root, lc, lane);
    // the symmetric sums count the member itself as a pair at r = 0 (once, in slice 0)
    constexpr bool kSelfPair = K::id == kKindHydro || K::id == kKindHydroAdj;
    lc.pairs += mem.n - ((kSelfPair && L.slice == 0 && mem.rank >= 0) ? 1 : 0);
    if constexpr (kLists) {
        // the member's slice-0 lane records its sub-list lengths, S and whether all fit
        int cnt4[4];
#pragma unroll
        for (int sl = 0; sl < 4; ++sl) {
            const int src = L.S > 1 ? sl * L.gw + (lane & (L.gw - 1)) : lane;
            const int v = __shfl_sync(0xffffffffu, mem.lcnt, (sl < L.S && src < 32) ? src : lane);
            cnt4[sl] = sl < L.S ? v : 0;
        }
        if (L.slice == 0 && mem.rank >= 0) {
            const int lsub = kListCap / L.S;
            const bool ok = cnt4[0] <= lsub && cnt4[1] <= lsub && cnt4[2] <= lsub && cnt4[3] <= lsub;
            a.o_lrec[entry] = make_int4(ok ? cnt4[0] | (cnt4[1] << 16) : 0, ok ? cnt4[2] | (cnt4[3] << 16) : 0, L.S,
                                        ok ? 1 : 0);
            a.o_lhw[entry] = rec[0].h * a.list_widen;
            a.o_lslot[mem.rank] = entry;
        }
    }
    slice_sum(mem, L);
    if (L.slice == 0 && mem.rank >= 0) write_result<MODE>(mem, a);
}

// One work item of the grouped kernels.  A group of more than 32 members is searched in
// parts of 32: one walk for all of them would pay every member a filter over the whole
// superset (at g = 64 on 4.2M clustered particles 15.5 ms a density pass, g = 128 more;
// in parts of 32 9.7 ms, all with the walk and staging before culling).
template <class K, int MODE>
__device__ __forceinline__ void process_group(const SearchArgs& a, WalkSmem& W, typename K::Tile& T, int gid,
                                              int nlarge, LocalCounters& lc, int lane) {
    const GroupDesc d = group_desc(a, gid, nlarge);
    if (d.cnt > 0) process_part<K, MODE>(a, W, T, d, lc, lane);
}

__device__ __forceinline__ int next_item(const SearchArgs& a, int lane, int take = 1) {
    int gid = 0;
    if (lane == 0) gid = atomicAdd(a.work, take);
    return __shfl_sync(0xffffffffu, gid, 0);
}

template <class K, int MODE>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, K::min_blocks) k_group(SearchArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    WalkSmem& W = reinterpret_cast<WalkSmem*>(smem_raw)[wib];
    clear_counters(W, lane);
    auto& T = reinterpret_cast<typename K::Tile*>(smem_raw + kWarpsPerBlock * sizeof(WalkSmem))[wib];
    LocalCounters lc;
    int nlarge;
    const int ng = group_count(a, nlarge);
    const int take = a.take;
    for (;;) {
        const int first = next_item(a, lane, take);
        if (first >= ng) break;
        for (int gid = first; gid < min(first + take, ng); ++gid)
            process_group<K, MODE>(a, W, T, gid, nlarge, lc, lane);
    }
    flush_counters(a, lc, W.ctr, lane);
}

// Two kinds of work item in one persistent queue: the groups of a0 (kind K0) first,
// then those of a1 (kind K1).  Both share the work counter of a0.
template <class K0, class K1>
__global__ void __launch_bounds__(kWarpsPerBlock * 32,
                                  K0::min_blocks < K1::min_blocks ? K0::min_blocks : K1::min_blocks)
k_group_pair(SearchArgs a0, SearchArgs a1) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr size_t kTileBytes = sizeof(typename K0::Tile) > sizeof(typename K1::Tile) ? sizeof(typename K0::Tile)
                                                                                        : sizeof(typename K1::Tile);
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    WalkSmem& W = reinterpret_cast<WalkSmem*>(smem_raw)[wib];
    clear_counters(W, lane);
    unsigned char* tile = smem_raw + kWarpsPerBlock * sizeof(WalkSmem) + wib * kTileBytes;
    LocalCounters lc;
    int large0, large1;
    const int n0 = group_count(a0, large0), n1 = group_count(a1, large1);
    for (;;) {
        const int gid = next_item(a0, lane);
        if (gid >= n0 + n1) break;
        if (gid < n0)
            process_group<K0, kAcc>(a0, W, *reinterpret_cast<typename K0::Tile*>(tile), gid, large0, lc,
                                    lane);
        else
            process_group<K1, kAcc>(a1, W, *reinterpret_cast<typename K1::Tile*>(tile), gid - n0, large1, lc, lane);
    }
    flush_counters(a0, lc, W.ctr, lane);
}

// The candidate superset of every group (inspection): the particles of the leaves that
// meet the sphere around the group centre covering every member's sphere, in walk order.
// Up to kSupSlots members per lane, one walk for the whole group.  FILL writes the
// candidates at x_off[group], else they are counted.
constexpr int kSupSlots = 4;

template <bool SYM, bool FILL>
__global__ void __launch_bounds__(kWarpsPerBlock * 32) k_superset(SearchArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    WalkSmem& W = reinterpret_cast<WalkSmem*>(smem_raw)[threadIdx.x >> 5];
    clear_counters(W, lane);
    LocalCounters lc;
    int nlarge;
    const int ng = group_count(a, nlarge);
    for (;;) {
        const int gid = next_item(a, lane);
        if (gid >= ng) break;
        const GroupDesc d = group_desc(a, gid, 0);
        MemberRec rec[kSupSlots];
#pragma unroll
        for (int mm = 0; mm < kSupSlots; ++mm) {
            const int k = lane + 32 * mm;
            rec[mm] = load_member(a, k < d.cnt ? a.U[d.base + k] : -1);
        }
        uint32_t cx = 0, cy = 0, cz = 0;
        if (!group_centre<kSupSlots>(a, rec, cx, cy, cz)) continue;
        // density: R_s = max_k (|m_k| + h_k); hydro: R_g = max_k |m_k|, hmax_g
        float rlane = 0.0f, hlane = 0.0f;
#pragma unroll
        for (int mm = 0; mm < kSupSlots; ++mm) {
            if (rec[mm].rank < 0) continue;
            const float mx = rel_coord(rec[mm].P.x, rec[mm].O.x, cx), my = rel_coord(rec[mm].P.y, rec[mm].O.y, cy),
                        mz = rel_coord(rec[mm].P.z, rec[mm].O.z, cz);
            const float mr = sqrtf(mx * mx + my * my + mz * mz);
            const float hf = (float)rec[mm].h;
            rlane = fmaxf(rlane, SYM ? mr : mr + 1.0f / (1.0f / hf));
            hlane = fmaxf(hlane, hf);
        }
        const float R = warp_max(rlane), hmax_g = warp_max(hlane);
        const float R2d = radius2_units(R);
        const float reach = SYM ? R + fmaxf(hmax_g, __uint_as_float(a.ncen[d.root].w)) : R;
        auto open_node = [&](bool have, const uint4& cen, const float4& ext, int) {
            const float R2 = SYM ? radius2_units(R + fmaxf(hmax_g, __uint_as_float(cen.w))) : R2d;
            return have && node_gap2(cen, ext, cx, cy, cz) <= R2;
        };
        Walk w = walk_begin();
        walk_visit(a, W, w, walk_start(a, d.root, cx, cy, cz, reach, lane), 0, lane, open_node);
        const int64_t pos = FILL ? a.x_off[gid] : 0;
        while (!w.empty() || w.total > w.done) {
            while (walk_can_step(a, w)) walk_step(a, W, w, 0, lane, open_node);
            walk_spill(a, W, w, lane);
            while (w.total > w.done) {
                const int64_t at = pos + w.done;
                int rank;
                const int nt = walk_take(W, w, lane, rank);
                if (FILL && lane < nt) {
                    if (at + lane < a.x_cap) a.x_idx[at + lane] = a.perm[rank];
                    else atomicOr(a.err, kErrCap);
                }
            }
        }
        if (lane == 0) W.ctr.cands += w.total;
        if (!FILL && lane == 0) a.x_cnt[gid] = w.total;
    }
    flush_counters(a, lc, W.ctr, lane);
}

// Density with the smoothing-length iteration inside the group (no host loop, no
// regrouping): after every walk + filter the members take the Newton / bisection step (in
// FP64); converged members leave the group, the centre and radius are recomputed over the
// remaining ones and the group walks again, until every member has converged or reached
// max_iter passes.  A particle's density at h depends only on the positions and its own
// h, so the iterates equal those of the pass-by-pass iteration (up to the order of the
// FP32 sums and the rounding of the step).
//
// Every lane takes its member's step, and an FP64 instruction of a warp takes 16 cycles of
// an SM: written with rho, dRho/dh and their divisions the step took about as long as a
// search.  In terms of the sums (see hsml_next) it has one division: N_eff = (32/3) S0 / m,
// g / g' = h (32 S0 - 3 N_ngb m) / (32 (3 S0 - S1)); the results, once per particle, two.
__device__ __forceinline__ bool hsml_step(const SearchArgs& a, const IterArgs& it, int r, float mf, double& h,
                                          double& lo, double& hi, float s0, float s1, int nngb, int pass,
                                          bool writer) {
    const double m = (double)mf, a0 = (double)s0;
    const double t = (32.0 / 3.0) * a0, nm = it.nngb * m;
    const double den = 3.0 * a0 - (double)s1;
    const bool done = fabs(t - nm) <= it.tol * m;
    if (done || pass >= it.max_iter) {
        if (writer) {
            const int orig = a.perm[r];
            const double ih = 1.0 / h;
            const double sigma = (8.0 / 3.14159265358979323846) * ih * ih * ih;
            it.rho[orig] = (float)(sigma * a0);
            it.drhodh[orig] = (float)(-sigma * ih * (double)s1);
            it.fgrad[orig] = (float)(3.0 * a0 / den);   // 1 / (1 + h / (3 rho) dRho/dh)
            it.nngb_out[orig] = nngb;
            if (it.iters) it.iters[orig] = pass;
            it.h_out[orig] = h;
            if (!done) atomicAdd(it.nfail, 1);
            if (it.max_pass) atomicMax(it.max_pass, pass);
        }
        return true;
    }
    if (t < nm) lo = h; else hi = h;
    double hn = h - h * ((t - nm) * 3.0 / (32.0 * den));
    if (!(hn > lo && hn < hi) || !isfinite(hn)) {
        const double cbrt2 = 1.2599210498948731647672106;
        if (isinf(hi)) hn = h * cbrt2;
        else if (lo == 0.0) hn = h / cbrt2;
        else hn = cbrt(0.5 * (lo * lo * lo + hi * hi * hi));
    }
    h = hn > it.h_max ? it.h_max : hn;   // (a NaN h stays one: it finds nothing)
    if (writer) {
        it.h64[r] = h;
        it.pfix[r].w = __float_as_uint((float)h);
    }
    return false;
}

__global__ void __launch_bounds__(kWarpsPerBlock * 32, 6) k_group_dens_iter(SearchArgs a, IterArgs it) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    WalkSmem& W = reinterpret_cast<WalkSmem*>(smem_raw)[wib];
    clear_counters(W, lane);
    PlainTile& T = reinterpret_cast<PlainTile*>(smem_raw + kWarpsPerBlock * sizeof(WalkSmem))[wib];
    LocalCounters lc;
    int nlarge;
    const int ng = group_count(a, nlarge);
    for (;;) {
        const int gid = next_item(a, lane);
        if (gid >= ng) break;
        const GroupDesc d = group_desc(a, gid, nlarge);
        if (d.cnt <= 0) continue;
        const Layout L = make_layout(d.cnt, lane, true, d.smax, false, PlainTile::cap);
        const int entry = member_entry(d, L, W, lane);
        MemberRec rec[1] = {load_member(a, L.k >= 0 ? a.U[entry] : -1)};
        double lo = 0.0, hi = __longlong_as_double(0x7ff0000000000000ll);
        if (lane == 0) W.ctr.walks++;
        for (int pass = 1;; ++pass) {
            uint32_t cx = 0, cy = 0, cz = 0;
            if (!group_centre<1>(a, rec, cx, cy, cz)) break;
            DMember mem;
            member_init(mem, a, rec[0], cx, cy, cz);
            group_search<KDens, kAcc>(a, W, T, L, mem, cx, cy, cz, d.root, lc, lane);
            lc.pairs += mem.n;
            slice_sum(mem, L);
            // every slice takes the step, from the sums of its member in slice 0
            const int src = max(L.k, 0);
            const float s0 = __shfl_sync(0xffffffffu, mem.s0 - mem.c0, src);
            const float s1 = __shfl_sync(0xffffffffu, mem.s1 - mem.c1, src);
            const int nn = __shfl_sync(0xffffffffu, mem.n, src);
            if (rec[0].rank >= 0 &&
                hsml_step(a, it, rec[0].rank, rec[0].O.w, rec[0].h, lo, hi, s0, s1, nn, pass, L.slice == 0))
                rec[0].rank = -1;
            // the new h (global memory) is read by the next pass's FP64 re-tests
            __syncwarp();
        }
    }
    flush_counters(a, lc, W.ctr, lane);
}

// ---------------------------------------------------------------------------------
// Individual form: one walk per particle.  The density and hydro loops take groups of one
// member in the kernel above: a warp walks for one particle, the box of its one member is
// a point, so the candidates kept are its neighbours, and its 32 lanes share them.
// One thread per particle with a depth-first walk (kept for the exports, which one lane
// writes) diverges at every node: 1.0M clustered particles, density + hydro 12.2 ms
// against 9.7 ms.
// ---------------------------------------------------------------------------------

template <int KIND, int MODE>
__global__ void __launch_bounds__(128) k_indiv(SearchArgs a) {
    const int lane = threadIdx.x & 31;
    LocalCounters lc;
    unsigned nodes = 0, cands = 0;
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < a.nu) {
        const int rank = a.U[u];
        const MemberRec rec = load_member(a, rank);
        const uint32_t cx = rec.P.x, cy = rec.P.y, cz = rec.P.z;
        DMember dm;
        HMember hm;
        float Rbox;
        if (KIND == 0) {
            member_init(dm, a, rec, cx, cy, cz);
            Rbox = (float)rec.h;
            if (MODE == kFill) dm.xpos = a.x_off[a.perm[rank]];
        } else {
            member_init(hm, a, rec, cx, cy, cz);
            Rbox = hm.h;
            if (MODE == kFill) hm.xpos = a.x_off[a.perm[rank]];
        }
        const float R2d = radius2_units(Rbox);
        int node = 0;
        while (node >= 0) {
            uint4 cen = a.ncen[node];
            float4 ext = a.next[node];
            int4 lk = a.nlink[node];
            nodes++;
            float gap2 = node_gap2(cen, ext, cx, cy, cz);
            float R2 = KIND == 0 ? R2d : radius2_units(fmaxf(Rbox, __uint_as_float(cen.w)));
            if (gap2 <= R2) {
                if (lk.z < 0) {
                    cands += lk.y;
                    lc.tests += lk.y;
                    for (int q = lk.x; q < lk.x + lk.y; ++q) {
                        uint4 Q = a.pfix[q];
                        float4 O = a.poff[q];
                        const float3 rel = make_float3(rel_coord(Q.x, O.x, cx), rel_coord(Q.y, O.y, cy),
                                                       rel_coord(Q.z, O.z, cz));
                        if (KIND == 0) {
                            dm.n++;
                            density_pair<MODE>(dm, a, rel, O.w, q, lc);
                        } else {
                            float hj = __uint_as_float(Q.w);
                            float dx = rel.x - hm.mx, dy = rel.y - hm.my, dz = rel.z - hm.mz;
                            float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                            float thr = fmaf(fmaxf(hm.h2, hj * hj), 1.0f + 3.0f * kBandRel, hm.bk);
                            if (r2 < thr) {
                                float4 H0 = a.hyd0[q], H1 = a.hyd1[q];
                                hm.n++;
                                hydro_pair<MODE>(hm, a, rel, make_float2(hj * hj, O.w), H0, H1, q, lc);
                            }
                        }
                    }
                    node = lk.w;
                } else {
                    node = lk.z;
                }
            } else {
                node = lk.w;
            }
        }
        lc.pairs += (KIND == 0) ? dm.n : hm.n - 1;
        if (KIND == 0) write_result<MODE>(dm, a);
        else write_result<MODE>(hm, a);
    }
    const unsigned long long tn = warp_sum(nodes), tc = warp_sum(cands);
    if (lane == 0) {
        atomicAdd(&a.ctr->nodes, tn);
        atomicAdd(&a.ctr->cands, tc);
    }
    flush_counters(a, lc, WalkCounters{0u, 0u, 0u, 0u}, lane);
}

// ---------------------------------------------------------------------------------
// Pieces of the searches that compute (count mode): one warp per window of up to 32
// consecutive work-list entries, whole chunks of g (g > 32: chunks of 32).  A chunk is cut
// (recursively) by the volume rule of k_split_groups, which cuts the exported groups: while
// its members' search sphere, ((sqrt(3)/2) box width + h_min)^3, exceeds split * (members)
// member spheres h_min^3, at the largest gap in key order between consecutive members (ties:
// nearest the middle; the middle when they are contiguous).  The pieces are not those groups:
// chunks are at most 32 and smaller on small lists, and every cut may be at a gap, where
// k_split_groups, which keeps a stack, halves a chunk after eight pending ranges.  In a batch,
// whose active particles are not runs, cuts are in the middle (gap cuts peel off single
// members there: a 16-box step 22.7 -> 23.5 ms).
//
// Pieces that reach far beyond their smallest h have the most candidates: they are stored
// from the end of the list downwards, and the search kernels take them first.
//
// The pieces go straight to the list, a block's together, with one atomic each for the
// large ones and the others: no scan of counts, and their number stays on the device.
// The list's order varies from run to run; every piece's sums are its own.
// ---------------------------------------------------------------------------------

constexpr int kCutWarps = 8;
constexpr float kLargeReach = 2.5f;  // 0.5 width + h_max above this many h_min: goes first

template <bool BATCH>
__global__ void __launch_bounds__(kCutWarps * 32) k_cut_pieces(CutArgs a) {
    __shared__ int cnt[2][kCutWarps];
    __shared__ int at[2];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // A forest that outgrew its arrays has only its roots: searched, every group would scan
    // its whole box, and the batch step, which reads nothing back, goes on until its end.
    if (BATCH && (*a.err & kErrNodes)) return;
    const int nwin = BATCH ? *a.nwindows_dev : a.nwindows;
    for (int w0 = blockIdx.x * kCutWarps; w0 < nwin; w0 += gridDim.x * kCutWarps) {   // block-uniform
        const int win = w0 + w;
        int base = 0, n = 0, g = a.g, root = 0, cfg = 0;
        float split = a.split;
        if (win < nwin) {
            if (BATCH) {
                const int4 C = a.windows[win];
                base = C.x;
                n = C.y;
                root = C.z;
                cfg = C.w;
                g = min(cfg & 0xff, 32);
                split = a.box_split[root];
            } else {
                base = win * a.width;
                n = min(a.width, a.nu - base);
            }
        }
        const int rank = lane < n ? a.U[base + lane] : -1;
        uint4 P = make_uint4(0u, 0u, 0u, 0u);
        float hf = 0.0f;
        if (rank >= 0) {
            P = a.pfix[rank];
            hf = (float)a.h64[rank];
        }
        const int up = __shfl_up_sync(0xffffffffu, rank, 1);
        uint32_t starts = __ballot_sync(0xffffffffu, lane % g == 0);
        uint32_t small = 0u, large = 0u;   // lane k: the mask of the k-th small / large piece
        int ns = 0, nl = 0;
        for (int s = 0; s < n;) {
            const uint32_t later = starts & ~((2u << s) - 1u);
            const int e = later ? min(__ffs(later) - 1, n) : n;
            const bool in = lane >= s && lane < e;
            float ext = 0.0f, hmin = 0.0f, hmax = 0.0f;
            if (e - s > 1) {
                const uint32_t x0 = __shfl_sync(0xffffffffu, P.x, s), y0 = __shfl_sync(0xffffffffu, P.y, s),
                               z0 = __shfl_sync(0xffffffffu, P.z, s);
                const int dx = in ? (int32_t)(P.x - x0) : 0, dy = in ? (int32_t)(P.y - y0) : 0,
                          dz = in ? (int32_t)(P.z - z0) : 0;
                const float wx = (float)((int64_t)__reduce_max_sync(0xffffffffu, dx) - __reduce_min_sync(0xffffffffu, dx)),
                            wy = (float)((int64_t)__reduce_max_sync(0xffffffffu, dy) - __reduce_min_sync(0xffffffffu, dy)),
                            wz = (float)((int64_t)__reduce_max_sync(0xffffffffu, dz) - __reduce_min_sync(0xffffffffu, dz));
                ext = fmaxf(wx, fmaxf(wy, wz)) * kUnitToBox;
                hmin = __uint_as_float(__reduce_min_sync(0xffffffffu, in ? __float_as_uint(hf) : 0x7f800000u));
                const float rel = fmaf(0.8660254f, ext / hmin, 1.0f);
                if (split > 0.0f && !(rel * rel * rel <= split * (float)(e - s))) {
                    const int mid = s + (e - s + 1) / 2;
                    const int gap = (in && lane > s) ? rank - up : 0;
                    const int best = BATCH ? 0 : __reduce_max_sync(0xffffffffu, gap);
                    int c = mid;
                    if (best > 1)
                        c = (int)(__reduce_min_sync(0xffffffffu, gap == best ? (unsigned)(abs(lane - mid) * 64 + lane)
                                                                             : 0xffffu) & 63u);
                    starts |= 1u << c;
                    continue;
                }
                hmax = warp_max(in ? hf : 0.0f);
            }
            const uint32_t piece = __ballot_sync(0xffffffffu, in);
            if (fmaf(0.5f, ext, hmax) > kLargeReach * hmin) {
                if (lane == nl) large = piece;
                ++nl;
            } else {
                if (lane == ns) small = piece;
                ++ns;
            }
            s = e;
        }
        if (lane == 0) {
            cnt[0][w] = ns;
            cnt[1][w] = nl;
        }
        __syncthreads();
        int pre[2] = {0, 0}, tot[2] = {0, 0};
        for (int k = 0; k < kCutWarps; ++k) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int v = cnt[q][k];
                if (k < w) pre[q] += v;
                tot[q] += v;
            }
        }
        if (threadIdx.x < 2 && tot[threadIdx.x] > 0) at[threadIdx.x] = atomicAdd(&a.npieces[threadIdx.x], tot[threadIdx.x]);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (lane >= (q ? nl : ns)) continue;
            const int64_t k = at[q] + pre[q] + lane;
            const int64_t slot = q ? a.cap - 1 - k : k;
            const uint32_t mask = q ? large : small;
            if (BATCH) a.pieces4[slot] = make_int4(base, (int)mask, root, cfg);
            else a.pieces[slot] = make_int2(base, (int)mask);
        }
        __syncthreads();   // cnt and at are rewritten by the next round
    }
}

int launch_cut_pieces(const CutArgs& a, int sm_count, cudaStream_t s) {
    cudaMemsetAsync(a.npieces, 0, 2 * sizeof(int), s);
    if (a.windows) {
        k_cut_pieces<true><<<8 * sm_count, kCutWarps * 32, 0, s>>>(a);
    } else {
        const int64_t blocks = std::min<int64_t>((a.nwindows + kCutWarps - 1) / kCutWarps, 32 * (int64_t)sm_count);
        if (blocks < 1) return SPHGRP_OK;
        k_cut_pieces<false><<<(unsigned)blocks, kCutWarps * 32, 0, s>>>(a);
    }
    note_launch();
    return check_cuda(cudaGetLastError(), "group pieces");
}

// ---------------------------------------------------------------------------------
// Grouping: chunks of g consecutive entries of the work list, each split (recursively)
// while the group's search sphere, ((sqrt(3)/2) box width + h_min)^3, exceeds split *
// (members) member spheres h_min^3.  The cut is at the largest gap in key order (see
// below).  A criterion on the walk's exact radius, max_k (|x_k - c| + h_k), against the
// smallest h split the same groups of the full workload but kept fewer members per walk
// on sparse active sets made of runs, 1.2-2x slower there at g >= 16.
// ---------------------------------------------------------------------------------

__global__ void k_split_groups(const int32_t* __restrict__ U, int nu, int g, float split,
                               const uint4* __restrict__ pfix, const double* __restrict__ h64,
                               int2* __restrict__ tmp, int32_t* __restrict__ cnt) {
    int ch = blockIdx.x * blockDim.x + threadIdx.x;
    int nch = (nu + g - 1) / g;
    if (ch >= nch) return;
    const int s0 = ch * g, e0 = min(s0 + g, nu);
    int2 st[16];
    int sp = 0, ng = 0;
    st[sp++] = make_int2(s0, e0);
    while (sp > 0) {
        int2 r = st[--sp];
        int s = r.x, e = r.y;
        bool keep = (e - s == 1) || split <= 0.0f;
        if (!keep) {
            uint4 P0 = pfix[U[s]];
            int lox = 0, loy = 0, loz = 0, hix = 0, hiy = 0, hiz = 0;
            float hmin = (float)h64[U[s]];
            for (int k = s + 1; k < e; ++k) {
                int rk = U[k];
                uint4 P = pfix[rk];
                int dx = (int32_t)(P.x - P0.x), dy = (int32_t)(P.y - P0.y), dz = (int32_t)(P.z - P0.z);
                lox = min(lox, dx); hix = max(hix, dx);
                loy = min(loy, dy); hiy = max(hiy, dy);
                loz = min(loz, dz); hiz = max(hiz, dz);
                hmin = fminf(hmin, (float)h64[rk]);
            }
            // search sphere of the group (box centre) relative to one member's sphere,
            // in volume: the candidates every member filters, per member's own
            const float ext = fmaxf(fmaxf((float)((int64_t)hix - lox), (float)((int64_t)hiy - loy)),
                                    (float)((int64_t)hiz - loz)) * kUnitToBox;
            const float rel = fmaf(0.8660254f, ext / hmin, 1.0f);
            keep = rel * rel * rel <= split * (float)(e - s);
        }
        if (keep) {
            tmp[s0 + ng++] = make_int2(s, e - s);
        } else {
            // Cut at the largest gap in key order (ties: the one nearest the middle): an
            // active set made of runs along the curve splits where one run ends and the
            // next begins; contiguous members split in the middle.  The stack holds one
            // pending range per level of the current path; gap cuts, which may peel one
            // member at a time, are taken while it holds fewer than 8, so that the
            // halving below them (at most log2(128) = 7 more levels) stays within 16.
            int mid = s + (e - s + 1) / 2;
            if (sp < 8) {
                int best = 1, bk = mid;
                for (int k = s + 1; k < e; ++k) {
                    const int gap = U[k] - U[k - 1];
                    if (gap > best || (gap == best && abs(k - mid) < abs(bk - mid))) {
                        best = gap;
                        bk = k;
                    }
                }
                mid = bk;
            }
            st[sp++] = make_int2(mid, e);
            st[sp++] = make_int2(s, mid);
        }
    }
    cnt[ch] = ng;
}

// Radius grouping (Sec. 2.1): a group starts at a work-list entry and takes the entries
// that follow while they lie closer than R = f h to its first particle (periodic
// minimum image), at most cap of them; the first entry farther away starts the next
// group.  One thread scans each run of kRadiusRun entries; groups go to tmp at the
// run's first entry.
__global__ void k_radius_groups(const int32_t* __restrict__ U, int nu, int cap, float f,
                                const uint4* __restrict__ pfix, const float4* __restrict__ poff,
                                const double* __restrict__ h64, int2* __restrict__ tmp, int32_t* __restrict__ cnt) {
    const int run = blockIdx.x * blockDim.x + threadIdx.x;
    const int s0 = run * kRadiusRun;
    if (s0 >= nu) return;
    const int e0 = min(s0 + kRadiusRun, nu);
    int ng = 0;
    int i = s0;
    while (i < e0) {
        const int r0 = U[i];
        const uint4 P0 = pfix[r0];
        const float4 O0 = poff[r0];
        const float R = f * (float)h64[r0];
        const float R2 = R * R;
        int j = i + 1;
        while (j < e0 && j - i < cap) {
            const int rj = U[j];
            const uint4 P = pfix[rj];
            const float4 O = poff[rj];
            const float dx = fix_diff(P.x, O.x, P0.x, O0.x);
            const float dy = fix_diff(P.y, O.y, P0.y, O0.y);
            const float dz = fix_diff(P.z, O.z, P0.z, O0.z);
            if (!(fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < R2)) break;
            ++j;
        }
        tmp[s0 + ng++] = make_int2(i, j - i);
        i = j;
    }
    cnt[run] = ng;
}

int launch_radius_groups(const int32_t* U, int nu, int cap, double f, const uint4* pfix, const float4* poff,
                         const double* h64, int2* tmp, int32_t* cnt, cudaStream_t s) {
    const int runs = (nu + kRadiusRun - 1) / kRadiusRun;
    k_radius_groups<<<blocks_for(runs, 64), 64, 0, s>>>(U, nu, cap, (float)f, pfix, poff, h64, tmp, cnt);
    note_launch();
    return check_cuda(cudaGetLastError(), "radius grouping");
}

__global__ void k_gather_groups(int nch, int g, const int2* __restrict__ tmp, const int32_t* __restrict__ cnt,
                                const int32_t* __restrict__ off, int2* __restrict__ groups) {
    int ch = blockIdx.x * blockDim.x + threadIdx.x;
    if (ch >= nch) return;
    int o = off[ch];
    for (int k = 0; k < cnt[ch]; ++k) groups[o + k] = tmp[ch * g + k];
}

int launch_split_groups(const int32_t* U, int nu, int g, float split, const uint4* pfix, const double* h64,
                        int2* tmp, int32_t* cnt, cudaStream_t s) {
    int nch = (nu + g - 1) / g;
    k_split_groups<<<blocks_for(nch, 128), 128, 0, s>>>(U, nu, g, split, pfix, h64, tmp, cnt);
    note_launch();
    return check_cuda(cudaGetLastError(), "group split");
}

int launch_gather_groups(int nch, int g, const int2* tmp, const int32_t* cnt, const int32_t* off, int2* groups,
                         cudaStream_t s) {
    k_gather_groups<<<blocks_for(nch, 256), 256, 0, s>>>(nch, g, tmp, cnt, off, groups);
    note_launch();
    return check_cuda(cudaGetLastError(), "group gather");
}

// ---------------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------------

// Shared memory of a block: below the 48 KB that a kernel may take on any device without an
// attribute of its own (attributes belong to a device; a flag per process would leave them
// unset on the next one).
constexpr size_t kPlainSmem = 48 * 1024;

template <class K>
constexpr size_t group_smem() {
    constexpr size_t sh = kWarpsPerBlock * (sizeof(WalkSmem) + sizeof(typename K::Tile));
    static_assert(sh <= kPlainSmem, "the kernel would need the opt-in attribute");
    return sh;
}

// Persistent grid: every resident block slot of the GPU, but at most one block per four
// groups (ngroups_host: their number, or a bound on it; -1: unknown).
template <typename Kern, typename... Args>
static int launch_persistent(Kern kern, size_t sh, int64_t ngroups_host, int sm_count, cudaStream_t s,
                             const char* what, Args... args) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWarpsPerBlock * 32, sh);
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)std::min(per_sm, kSpillWarpsPerSM / kWarpsPerBlock) * sm_count;
    if (ngroups_host >= 0) grid = std::min<int64_t>(grid, (ngroups_host + kWarpsPerBlock - 1) / kWarpsPerBlock);
    if (grid < 1) grid = 1;
    kern<<<(unsigned)grid, kWarpsPerBlock * 32, sh, s>>>(args...);
    note_launch();
    return check_cuda(cudaGetLastError(), what);
}

// Items are numbered by an int, and a listed group of more than 32 members is up to four of
// them: more than kMaxItems go in several launches (the radius and tree modes on more than
// 2^29 particles).
constexpr int kMaxItems = 0x7fffffff - (1 << 20);   // less what the warps take past the end

template <class Launch>
static int launch_items(const SearchArgs& a, cudaStream_t s, Launch launch) {
    const int most = kMaxItems / a.parts;
    if (!a.groups || a.ngroups <= most) return launch(a);
    int rc = SPHGRP_OK;
    for (int off = 0; off < a.ngroups && !rc; off += most) {
        SearchArgs b = a;
        b.groups = a.groups + off;
        b.ngroups = std::min(most, a.ngroups - off);
        if (off > 0) cudaMemsetAsync(a.work, 0, sizeof(int), s);
        rc = launch(b);
    }
    return rc;
}

template <class K, int MODE>
static int launch_group(const SearchArgs& a, int sm_count, cudaStream_t s) {
    if (a.g > 128) return set_error(SPHGRP_EINVAL, "group_size must be <= 128");
    SearchArgs b = a;
    b.parts = (a.g + kPartMax - 1) / kPartMax;
    // many single members: several items per counter access (one address serves all warps)
    b.take = a.g == 1 && a.ngroups >= 1 << 16 ? 4 : 1;
    return launch_items(b, s, [&](const SearchArgs& c) {
        return launch_persistent(k_group<K, MODE>, group_smem<K>(),
                                 c.npieces ? c.nu : (int64_t)c.ngroups * c.parts, sm_count, s, "grouped search kernel", c);
    });
}

template <bool SYM, bool FILL>
static int launch_superset(const SearchArgs& a, int sm_count, cudaStream_t s) {
    if (a.g > 32 * kSupSlots) return set_error(SPHGRP_EINVAL, "group_size must be <= 128");
    return launch_persistent(k_superset<SYM, FILL>, kWarpsPerBlock * sizeof(WalkSmem), a.ngroups, sm_count, s,
                             "superset kernel", a);
}

template <class K>
static int launch_group_k(const SearchArgs& a, int mode, int sm_count, cudaStream_t s) {
    switch (mode) {
        case kAcc: return launch_group<K, kAcc>(a, sm_count, s);
        case kCount: return launch_group<K, kCount>(a, sm_count, s);
        case kFill: return launch_group<K, kFill>(a, sm_count, s);
        case kSupCount: return launch_superset<K::sym, false>(a, sm_count, s);
        case kSupFill: return launch_superset<K::sym, true>(a, sm_count, s);
    }
    return set_error(SPHGRP_EINVAL, "bad search mode");
}

int launch_search_dev(const SearchArgs& a, int kind, int max_g, int sm_count, cudaStream_t s) {
    if (max_g < 1 || max_g > 128) return set_error(SPHGRP_EINVAL, "group size outside [1, 128]");
    cudaMemsetAsync(a.work, 0, sizeof(int), s);
    SearchArgs b = a;
    b.g = max_g;   // bound only; the pieces carry their members
    switch (kind) {
        case kKindDensity:
            return b.o_s2 ? launch_group<KDens2, kAcc>(b, sm_count, s) : launch_group<KDens, kAcc>(b, sm_count, s);
        case kKindHydro: return launch_group<KHydro, kAcc>(b, sm_count, s);
        case kKindHydroAdj: return launch_group<KHAdj, kAcc>(b, sm_count, s);
        case kKindDensityAdj: return launch_group<KDAdj, kAcc>(b, sm_count, s);
    }
    return set_error(SPHGRP_EINVAL, "bad kind");
}

int launch_density_iter(const SearchArgs& a, const IterArgs& it, int max_g, int sm_count, cudaStream_t s) {
    if (max_g < 1 || max_g > 128) return set_error(SPHGRP_EINVAL, "group size outside [1, 128]");
    cudaMemsetAsync(a.work, 0, sizeof(int), s);
    SearchArgs b = a;
    b.parts = (a.g + kPartMax - 1) / kPartMax;
    return launch_items(b, s, [&](const SearchArgs& c) {
        return launch_persistent(k_group_dens_iter, group_smem<KDens>(),
                                 c.npieces ? c.nu : (int64_t)c.ngroups * c.parts, sm_count, s,
                                 "grouped density iteration kernel", c, it);
    });
}

template <class K0, class K1>
static int launch_pair(const SearchArgs& a0, const SearchArgs& a1, int sm_count, cudaStream_t s) {
    constexpr size_t tile = sizeof(typename K0::Tile) > sizeof(typename K1::Tile) ? sizeof(typename K0::Tile)
                                                                                  : sizeof(typename K1::Tile);
    constexpr size_t sh = kWarpsPerBlock * (sizeof(WalkSmem) + tile);
    static_assert(sh <= kPlainSmem, "the kernel would need the opt-in attribute");
    return launch_persistent(k_group_pair<K0, K1>, sh, -1, sm_count, s, "paired search kernel", a0, a1);
}

int launch_search_pair(const SearchArgs& a0, int kind0, const SearchArgs& a1, int kind1, int max_g, int sm_count,
                       cudaStream_t s) {
    if (max_g < 1 || max_g > 128) return set_error(SPHGRP_EINVAL, "group size outside [1, 128]");
    cudaMemsetAsync(a0.work, 0, sizeof(int), s);
    if (kind0 == kKindHydro && kind1 == kKindHydroAdj) return launch_pair<KHydro, KHAdj>(a0, a1, sm_count, s);
    return set_error(SPHGRP_EINVAL, "unsupported kind pair");
}

int launch_search(const SearchArgs& a, int kind, int mode, bool grouped, int sm_count, cudaStream_t s) {
    if (a.nu <= 0) return SPHGRP_OK;
    if (grouped) {
        cudaMemsetAsync(a.work, 0, sizeof(int), s);
        switch (kind) {
            case 0:
                if (mode == kAcc && a.o_s2) return launch_group<KDens2, kAcc>(a, sm_count, s);
                return launch_group_k<KDens>(a, mode, sm_count, s);
            case 1: return launch_group_k<KHydro>(a, mode, sm_count, s);
            case 2:
                if (mode != kAcc) return set_error(SPHGRP_EINVAL, "adjoint kernels accumulate only");
                return launch_group<KHAdj, kAcc>(a, sm_count, s);
            case 3:
                if (mode != kAcc) return set_error(SPHGRP_EINVAL, "adjoint kernels accumulate only");
                return launch_group<KDAdj, kAcc>(a, sm_count, s);
            case kKindVelocity:
                if (mode != kAcc) return set_error(SPHGRP_EINVAL, "the velocity derivatives accumulate only");
                return launch_group<KVel, kAcc>(a, sm_count, s);
            case kKindDensityVel:
                if (mode != kAcc) return set_error(SPHGRP_EINVAL, "velocity derivatives accumulate only");
                return launch_group<KDensVel, kAcc>(a, sm_count, s);
            case kKindDensityList:
                if (mode != kAcc || a.g > 32)
                    return set_error(SPHGRP_EINVAL, "candidate lists: accumulation, group size <= 32");
                return launch_group<KDensList, kAcc>(a, sm_count, s);
        }
        return set_error(SPHGRP_EINVAL, "bad kind");
    }
    if (kind != 0 && kind != 1)
        return set_error(SPHGRP_EINVAL, "the adjoint kernels exist in the grouped form only");
    if (mode == kAcc) {
        // one walk per particle, a warp to a particle: groups of one member
        cudaMemsetAsync(a.work, 0, sizeof(int), s);
        SearchArgs b = a;
        b.g = 1;
        b.ngroups = a.nu;
        return kind == 0 ? launch_group<KDens, kAcc>(b, sm_count, s) : launch_group<KHydro, kAcc>(b, sm_count, s);
    }
    const int blocks = blocks_for(a.nu, 128);
    if (kind == 0 && mode == kCount) k_indiv<0, kCount><<<blocks, 128, 0, s>>>(a);
    else if (kind == 0 && mode == kFill) k_indiv<0, kFill><<<blocks, 128, 0, s>>>(a);
    else if (kind == 1 && mode == kCount) k_indiv<1, kCount><<<blocks, 128, 0, s>>>(a);
    else if (kind == 1 && mode == kFill) k_indiv<1, kFill><<<blocks, 128, 0, s>>>(a);
    else return set_error(SPHGRP_EINVAL, "bad search mode");
    note_launch();
    return check_cuda(cudaGetLastError(), "individual search kernel");
}

// ---------------------------------------------------------------------------------
// Smoothing-length iteration: per unconverged particle, FP64
// ---------------------------------------------------------------------------------

// One particle's step of the smoothing-length iteration from its density sums at h
// (S0 = sum m w, S1 = sum m (q w' + 3 w)) after `pass` passes.  With rho = sigma S0,
// dRho/dh = -(sigma / h) S1 and sigma = 8 / (pi h^3), the quantities of the iteration
// reduce to the sums themselves:
//   N_eff = (4 pi / 3) h^3 rho / m = (32 / 3) S0 / m,
//   f = 1 / (1 + h / (3 rho) dRho/dh) = 3 S0 / (3 S0 - S1),
//   g / g' = h (32 S0 - 3 N_ngb m) / (32 (3 S0 - S1))  (the Newton step).
// The convergence test |N_eff - N_ngb| <= tol is taken in FP64, as
// |(32/3) S0 - N_ngb m| <= tol m (no division); the sums themselves are FP32, so the
// Newton step and the bisection of the bracket carry no more than FP32 accuracy either
// and are taken in FP32 (FP64 division is slow on this part and would buy nothing).
// finish: converged (or no iteration asked), or the last pass; else hn is the next h and
// [lo, hi) the updated bracket (opened at pass 1).
struct HsmlStep {
    bool finish, converged;
    double hn;
};

__device__ __forceinline__ HsmlStep hsml_next(double h, float m, float s0, float s1, double nngb, double tol,
                                              bool iterate, int pass, int max_iter, double& lo, double& hi) {
    HsmlStep o;
    const double t = (32.0 / 3.0) * (double)s0, nm = nngb * (double)m;
    o.converged = !iterate || fabs(t - nm) <= tol * (double)m;
    o.finish = o.converged || pass >= max_iter;
    o.hn = h;
    if (o.finish) return o;
    if (pass == 1) {
        lo = 0.0;
        hi = __longlong_as_double(0x7ff0000000000000ll);
    }
    if (t < nm) lo = h; else hi = h;
    const float hf = (float)h;
    const float num = fmaf(-3.0f * (float)nngb, m, 32.0f * s0);
    const float den = 32.0f * (3.0f * s0 - s1);
    double hn = (double)(hf - hf * (num / den));
    if (!(hn > lo && hn < hi) || !isfinite(hn)) {
        // volume bisection of the bracket
        if (isinf(hi)) hn = (double)(hf * 1.25992104989487316f);
        else if (lo == 0.0) hn = (double)(hf * 0.79370052598409974f);
        else {
            const float l = (float)lo, u = (float)hi;
            hn = (double)cbrtf(0.5f * (l * l * l + u * u * u));
        }
    }
    o.hn = hn;
    return o;
}


// One particle's pass of the smoothing-length iteration: u = its work-list entry, r its
// rank, s0 / s1 / n its density sums at the current h.  Runs as its own kernel with one
// particle per thread: in the search kernel's epilogue only one slice of each warp would
// hold the members, which doubles the FP64 issue.
__device__ __forceinline__ void hsml_update(const UpdateArgs& a, int u, int r, float s0f, float s1f, int n) {
    const double h = a.h64[r];
    const float m = a.poff[r].w;
    const int pass = a.npass ? a.npass[r] + 1 : a.it;
    if (a.npass) a.npass[r] = pass;
    double lo = pass == 1 ? 0.0 : a.lo[r];
    double hi = pass == 1 ? __longlong_as_double(0x7ff0000000000000ll) : a.hi[r];
    const HsmlStep st = hsml_next(h, m, s0f, s1f, a.nngb, a.tol, a.iterate != 0, pass, a.max_iter, lo, hi);
    if (st.finish) {
        if (a.res_k) {
            a.res_k[r] = make_float4(s0f, s1f, __int_as_float(n), __int_as_float(pass));
        } else {
            hsml_write(a.perm[r], h, s0f, s1f, n, pass, a.h_out, a.rho, a.drhodh, a.fgrad, a.nngb_out, a.iters);
        }
        if (a.vsum && !a.res_k) {
            // div v = -(1/rho) sum m v_ij . grad W, curl v = (1/rho) sum m v_ij x grad W
            const int orig = a.perm[r];
            const float hf = (float)h;
            const float rinv = hf * hf * hf / (2.54647908947032537f * s0f);   // 1 / rho
            const float4 V = a.vsum[r];
            a.divv[orig] = V.x * rinv;
            a.curlv[3 * (int64_t)orig] = V.y * rinv;
            a.curlv[3 * (int64_t)orig + 1] = V.z * rinv;
            a.curlv[3 * (int64_t)orig + 2] = V.w * rinv;
        }
        a.keep[u] = 0;
        if (!st.converged) atomicAdd(a.nfail, 1);
        return;
    }
    a.lo[r] = lo;
    a.hi[r] = hi;
    a.h64[r] = st.hn;
    a.pfix[r].w = __float_as_uint((float)st.hn);
    a.keep[u] = 1;
}

__global__ void k_hsml_update(UpdateArgs a) {
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= a.nu) return;
    const int r = a.U[u];
    hsml_update(a, u, r, a.s0[r], a.s1[r], a.n[r]);
}

// Passes 2, 3, ... of the recycled iteration, one thread per unconverged particle: while
// its h stays within the widened radius h_w of its pass-1 candidate list, the density
// sums at h are those of the list's members inside h (the list holds every particle
// within h_w), so the particle iterates on its own list without a tree walk.  The
// decisions are the exact ones of the grouped kernel (FP32 on exact fixed-point
// differences, FP64 re-test in the band).  A particle whose h leaves h_w, or whose list
// overflowed, is flagged for a walk pass (keep = 1) with its iterate and bracket stored.
__global__ void __launch_bounds__(128) k_list_iterate(ListIterArgs a) {
    const int lane = threadIdx.x & 31;
    LocalCounters lc;
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < a.nu) {
        const int r = a.U[u];
        const int slot = a.lslot[r];
        const int4 rec = a.lrec[slot];
        const double hw = a.lhw[slot];
        int pass = a.npass[r];
        double h = a.h64[r], lo = a.lo[r], hi = a.hi[r];
        const uint4 P = a.pfix_in[r];
        const float4 O = a.poff[r];
        const float m = O.w;
        bool walk = rec.w == 0;
        while (!walk) {
            if (!(h <= hw)) {
                walk = true;
                break;
            }
            ++pass;
            const float hf = (float)h;
            const float h2 = (float)(h * h);
            const float h2lo = h2 * (1.0f - 3.0f * kBandRel), h2hi = h2 * (1.0f + 3.0f * kBandRel);
            const float hinv = 1.0f / hf;
            const double hh = __dmul_rn(h, h);
            const int lsub = kListCap / rec.z;
            float S0 = 0.0f, C0 = 0.0f, S1 = 0.0f, C1 = 0.0f, p0 = 0.0f, p1 = 0.0f;
            int n = 0;
            for (int sl = 0; sl < rec.z; ++sl) {
                const int cnt = sl == 0 ? (rec.x & 0xffff) : sl == 1 ? (rec.x >> 16) : sl == 2 ? (rec.y & 0xffff)
                                                                                               : (rec.y >> 16);
                // sub-lists start at multiples of 4 entries (kListCap / S, S in {1, 2, 4}):
                // four entries per step, read as one int4 and gathered together, so that a
                // thread keeps eight candidate loads in flight
                const int4* L4 = reinterpret_cast<const int4*>(a.list + (int64_t)slot * kListCap + sl * lsub);
                for (int k0 = 0; k0 < cnt; k0 += 4) {
                    const int4 J4 = L4[k0 >> 2];
                    const int jj[4] = {J4.x, J4.y, J4.z, J4.w};
                    uint4 Q[4];
                    float4 Oj[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (k0 + e < cnt) {
                            Q[e] = __ldg(a.pfix_in + jj[e]);
                            Oj[e] = __ldg(a.poff + jj[e]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (k0 + e >= cnt) break;
                        const float dx = fix_diff(Q[e].x, Oj[e].x, P.x, O.x);
                        const float dy = fix_diff(Q[e].y, Oj[e].y, P.y, O.y);
                        const float dz = fix_diff(Q[e].z, Oj[e].z, P.z, O.z);
                        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                        bool in = r2 < h2lo;
                        if (!in && r2 < h2hi) {
                            in = exact_r2(a.xd, a.yd, a.zd, r, jj[e]) < hh;
                            lc.retests++;
                        }
                        if (!in) continue;
                        ++n;
                        const float q = r2 * rsqrtf(fmaxf(r2, 1.0e-30f)) * hinv;
                        float w, dw;
                        m4_shape(q, w, dw);
                        p0 = fmaf(Oj[e].w, w, p0);
                        p1 = fmaf(Oj[e].w, fmaf(q, dw, 3.0f * w), p1);
                    }
                    if ((k0 & 15) == 12) {
                        kahan_add(S0, C0, p0);
                        kahan_add(S1, C1, p1);
                        p0 = p1 = 0.0f;
                    }
                }
            }
            kahan_add(S0, C0, p0);
            kahan_add(S1, C1, p1);
            lc.pairs += n;
            const float s0 = S0 - C0, s1 = S1 - C1;
            const HsmlStep st = hsml_next(h, m, s0, s1, a.nngb, a.tol, true, pass, a.max_iter, lo, hi);
            if (st.finish) {
                hsml_write(a.perm[r], h, s0, s1, n, pass, a.h_out, a.rho, a.drhodh, a.fgrad, a.nngb_out, a.iters);
                if (!st.converged) atomicAdd(a.nfail, 1);
                break;
            }
            h = st.hn;
        }
        // (positions are read through the read-only path: pfix is not written here; its
        // FP32 copy of h is not read during the density call, and the hydro and velocity
        // entry points rewrite it from the caller's h)
        a.keep[u] = walk ? 1 : 0;
        a.npass[r] = pass;
        a.h64[r] = h;
        a.lo[r] = lo;
        a.hi[r] = hi;
    }
    // only pairs and re-tests are counted: the lists are not tree-search candidates
    int mp = u < a.nu ? a.npass[a.U[u]] : 0;
    for (int o = 16; o > 0; o >>= 1) {
        lc.pairs += __shfl_xor_sync(0xffffffffu, lc.pairs, o);
        lc.retests += __shfl_xor_sync(0xffffffffu, lc.retests, o);
        mp = max(mp, __shfl_xor_sync(0xffffffffu, mp, o));
    }
    if (lane == 0) {
        if (lc.pairs) atomicAdd(&a.ctr->pairs, lc.pairs);
        if (lc.retests) atomicAdd(&a.ctr->retests, lc.retests);
        if (a.max_pass) atomicMax(a.max_pass, mp);
    }
}

int launch_list_iterate(const ListIterArgs& a, cudaStream_t s) {
    if (a.nu <= 0) return SPHGRP_OK;
    // no shared memory: all of it as L1, which holds the candidates that neighbouring
    // particles gather (set on each call: the attribute belongs to the current device)
    int rc = check_cuda(cudaFuncSetAttribute(k_list_iterate, cudaFuncAttributePreferredSharedMemoryCarveout, 0),
                        "list iteration");
    if (rc) return rc;
    k_list_iterate<<<blocks_for(a.nu, 128), 128, 0, s>>>(a);
    note_launch();
    return check_cuda(cudaGetLastError(), "list iteration");
}

int launch_hsml_update(const UpdateArgs& a, cudaStream_t s) {
    if (a.nu <= 0) return SPHGRP_OK;
    k_hsml_update<<<blocks_for(a.nu, 256), 256, 0, s>>>(a);
    note_launch();
    return check_cuda(cudaGetLastError(), "hsml update");
}

}  // namespace sphgrp
