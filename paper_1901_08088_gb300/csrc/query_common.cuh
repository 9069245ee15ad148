// Device code shared by the traversals (query.cu: rope walks of the binary
// tree, query_wide.cu: walk of the 32-wide boxes): tree loads, list stores,
// the exact pair decision, periodic images.  The decision and the image
// argument are set out at the top of query.cu.
#pragma once

#include "qbvh_internal.cuh"

namespace qbvh {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

// Read-only loads of tree words (nodes, leaves).  QBVH_TREE_EVICT_LAST = 1
// marks them evict-last in L2, so that list writes streaming through L2 evict
// them after everything else.  That paid while the list went out as 4-byte
// stores (1.4 GB of DRAM writes per launch at N = 2M: query 1.92 -> 1.84 ms);
// with whole-sector row writes (1.0 GB) plain loads are faster (10-bit nodes
// 1.266 -> 1.240 ms, FP32 nodes 1.243 -> 1.237 ms), so it is off.
// QBVH_NODE_V8 = 1 reads a 32-byte FP32 node with one 256-bit load (sm_100
// and later) instead of two 128-bit ones (same speed, one instruction).
#ifndef QBVH_TREE_EVICT_LAST
#define QBVH_TREE_EVICT_LAST 0
#endif
#ifndef QBVH_NODE_V8
#define QBVH_NODE_V8 1
#endif
__device__ __forceinline__ float4 tree_ld(const float4 *p)
{
#if QBVH_TREE_EVICT_LAST
    unsigned long long pol;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    float4 v;
    asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "l"(pol));
    return v;
#else
    return __ldg(p);
#endif
}
__device__ __forceinline__ int4 tree_ld(const int4 *p)
{
#if QBVH_TREE_EVICT_LAST
    unsigned long long pol;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    int4 v;
    asm("ld.global.nc.L2::cache_hint.v4.s32 {%0, %1, %2, %3}, [%4], %5;"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
    return v;
#else
    return __ldg(p);
#endif
}
// both halves of a 32-byte FP32 node (32-byte aligned: node arrays come from
// the allocator's 256-byte aligned blocks)
__device__ __forceinline__ void node32_ld(const float4 *p, float4 &a, float4 &b)
{
#if QBVH_NODE_V8 && QBVH_TREE_EVICT_LAST
    asm("ld.global.nc.L2::evict_last.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w) : "l"(p));
#elif QBVH_NODE_V8
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w) : "l"(p));
#else
    a = tree_ld(p);
    b = tree_ld(p + 1);
#endif
}

// Store of one list entry.  QBVH_ROW_STORE: 0 = streaming (evict-first),
// 1 = cache at L2 (.cg), 2 = default write-back.
#ifndef QBVH_ROW_STORE
#define QBVH_ROW_STORE 0
#endif
__device__ __forceinline__ void row_store(int *p, int v)
{
#if QBVH_ROW_STORE == 0
    __stcs(p, v);
#elif QBVH_ROW_STORE == 1
    __stcg(p, v);
#else
    *p = v;
#endif
}

// One whole sector: 8 entries, dst on a 32-byte boundary, entry k at ring[32 k].
// The lanes of a warp write to 32 rows, and L1 takes a cycle per row and
// instruction, so one 32-byte store (sm_100 and later) takes half the cycles of two
// 16-byte ones.
__device__ __forceinline__ void store_sector(int *dst, const int *ring)
{
    asm volatile("st.global.cs.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(ring[0]), "r"(ring[32]),
                 "r"(ring[64]), "r"(ring[96]), "r"(ring[128]), "r"(ring[160]), "r"(ring[192]), "r"(ring[224])
                 : "memory");
}

struct Query {
    float xi, yi, zi;     // own position
    int self;             // own sorted index
    int self_id;          // own original index
    float nLx, nLy, nLz;  // image shift n L
    float px, py, pz;     // image centre fl(x_i + n L)
    float rl2;
    float rl2_lo, rl2_hi; // double-precision data: band of the FP32 test around rl2
    int pair;             // double-precision data: type pair of the current tree
    // Lennard-Jones value of an image pair (fused option): per axis the
    // difference fl(fl(xj - v1) - v2), the once-rounded x_j - x_i - n L
    float vx1, vy1, vz1, vx2, vy2, vz2;
};

// d2 of the exact test (see the header comment) for leaf position q.
// SHIFT = false is the zero image, where subtracting n L = 0 is the identity.
template <bool SHIFT>
__device__ __forceinline__ float exact_d2(const Query &c, const float4 q)
{
#if QBVH_F32X2
    f32x2 dxy = f2_sub(f2_pack(q.x, q.y), f2_pack(c.xi, c.yi));
    float dz = __fsub_rn(q.z, c.zi);
    if (SHIFT) {
        dxy = f2_sub(dxy, f2_pack(c.nLx, c.nLy));
        dz = __fsub_rn(dz, c.nLz);
    }
    float sx, sy;
    f2_unpack(f2_mul(dxy, dxy), sx, sy);
    return __fadd_rn(__fadd_rn(sx, sy), __fmul_rn(dz, dz));
#else
    float dx = __fsub_rn(q.x, c.xi);
    float dy = __fsub_rn(q.y, c.yi);
    float dz = __fsub_rn(q.z, c.zi);
    if (SHIFT) {
        dx = __fsub_rn(dx, c.nLx);
        dy = __fsub_rn(dy, c.nLy);
        dz = __fsub_rn(dz, c.nLz);
    }
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
#endif
}

// Double-precision particle data (Sec. 2.2).  The list's decision is the
// pinned FP64 expression
//   dx = fl(xj - xi); dx = fl(dx - L rint(fl(dx Linv))), same for y, z,
//   d2 = fl(fl(fl(dx^2) + fl(dy^2)) + fl(dz^2)) < fl(r^2),
// taken under the walk's image without rint, as in FP32 (the argument in the
// header comment holds with the FP64 unit roundoff).  The leaf words hold
// the positions rounded to FP32, and the FP32 d2 of those decides whenever
// it lies outside [rl2_lo, rl2_hi]: the host sets that band from a bound on
// the difference of the two computations for pairs within the radius
// (per component at most 2^-21 L, see qbvh_query), so it cannot change a
// decision.  Inside the band the FP64 positions decide.
template <bool SHIFT>
__device__ __forceinline__ double exact_d2_64(const QueryArgs &A, const Query &c, int j)
{
    const double2 *pj = reinterpret_cast<const double2 *>(A.leaves64 + j);
    const double2 *pi = reinterpret_cast<const double2 *>(A.leaves64 + c.self);
    const double2 jxy = __ldg(pj), jz = __ldg(pj + 1), ixy = __ldg(pi), iz = __ldg(pi + 1);
    double dx = __dsub_rn(jxy.x, ixy.x);
    double dy = __dsub_rn(jxy.y, ixy.y);
    double dz = __dsub_rn(jz.x, iz.x);
    if (SHIFT) {
        const double L = A.L64;
        if (c.nLx != 0.f) dx = __dsub_rn(dx, c.nLx > 0.f ? L : -L);
        if (c.nLy != 0.f) dy = __dsub_rn(dy, c.nLy > 0.f ? L : -L);
        if (c.nLz != 0.f) dz = __dsub_rn(dz, c.nLz > 0.f ? L : -L);
    }
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// 27-bit set of the periodic images whose padded search sphere overlaps the
// root AABB of a tree (Sec. 2.3): bit 9 (nx+1) + 3 (ny+1) + (nz+1).
__device__ __forceinline__ unsigned image_mask(float x, float y, float z, float L, const SegInfo &g, float rs2)
{
    float gap[3][3];
    const float xs[3] = {x, y, z};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const float p = (m == 1) ? xs[d] : __fadd_rn(xs[d], (m == 0) ? -L : L);
            gap[d][m] = fmaxf(fmaxf(__fsub_rd(g.rlo[d], p), __fsub_rd(p, g.rhi[d])), 0.f);
        }
    }
    unsigned mask = 0u;
#pragma unroll
    for (int mx = 0; mx < 3; ++mx)
#pragma unroll
        for (int my = 0; my < 3; ++my)
#pragma unroll
            for (int mz = 0; mz < 3; ++mz) {
                const float d2 = __fmaf_rd(gap[0][mx], gap[0][mx],
                                           __fmaf_rd(gap[1][my], gap[1][my], __fmul_rd(gap[2][mz], gap[2][mz])));
                if (d2 <= rs2) mask |= 1u << (mx * 9 + my * 3 + mz);
            }
    return mask;
}

__device__ __forceinline__ void set_image(Query &c, int img, float L)
{
    const int nx = img / 9 - 1, ny = (img / 3) % 3 - 1, nz = img % 3 - 1;
    c.nLx = nx == 0 ? 0.f : (nx > 0 ? L : -L);
    c.nLy = ny == 0 ? 0.f : (ny > 0 ? L : -L);
    c.nLz = nz == 0 ? 0.f : (nz > 0 ? L : -L);
    c.px = nx == 0 ? c.xi : __fadd_rn(c.xi, c.nLx);
    c.py = ny == 0 ? c.yi : __fadd_rn(c.yi, c.nLy);
    c.pz = nz == 0 ? c.zi : __fadd_rn(c.zi, c.nLz);
}

template <bool WIDE>
__device__ __forceinline__ int seg_of_sorted(const QueryArgs &a, int s)
{
    if (WIDE) return (int)(__ldg(reinterpret_cast<const unsigned long long *>(a.keys_sorted) + s) >> 30);
    if (a.n_types > 1) return (int)(__ldg(reinterpret_cast<const unsigned *>(a.keys_sorted) + s) >> 30);
    return 0;
}

// Largest row count: one atomic per warp, skipped when it cannot raise the maximum.
__device__ __forceinline__ void warp_max_count(int my_count, DevStatus *status)
{
    const int m = __reduce_max_sync(FULL, my_count);
    if ((threadIdx.x & 31) == 0 && m > 0 && m > __ldcg(&status->max_count)) atomicMax(&status->max_count, m);
}

// ---- sparse trees: one particle per warp ---------------------------------
// A tree of few, widely spaced particles (the large spheres of a
// size-asymmetric mixture) makes poor packets: 32 consecutive Z-order
// particles then span much of the box, so a packet walk is 32 separate
// walks run one after another on one warp, and the few such warps end long
// after the rest (mixture L = 100: the 400 large particles' walks of the
// small-particle tree took 1.5 ms against 0.55 ms for all small-small
// pairs).  Tree `ta` of a single-system FP32 build of 2 to 4 types (32-bit
// keys) is walked one particle per warp instead when it holds at most
// QBVH_SPARSE_MAX particles and a packet of 32 spans more than twice its
// largest list radius:
// 32 L^3 / count > (2 r_max)^3.  The choice changes only which warp walks a
// particle: the walk visits the same nodes and leaves in the same order, so
// rows are the same either way.
#ifndef QBVH_SPARSE_TREES
#define QBVH_SPARSE_TREES 1
#endif
#ifndef QBVH_SPARSE_MAX
#define QBVH_SPARSE_MAX 4096
#endif
__device__ __forceinline__ bool sparse_tree(const QueryArgs &a, int ta)
{
    const int count = a.seg[ta].count;
    if (count == 0 || count > QBVH_SPARSE_MAX) return false;
    const int T = a.n_types;
    float r = 0.f;
    for (int tb = 0; tb < T; ++tb) r = fmaxf(r, a.r_list[ta * T + tb]);
    const float L = a.sys[0].L, d = 2.f * r;
    return 32.f * L * L * L > (float)count * d * d * d;
}

}  // namespace

// SM count of the current device, looked up once per device (the value
// only sizes the sparse-tree blocks: a stale or racing read costs speed, not
// correctness; the table is written once per slot with the same value)
static inline int sm_count_current()
{
    constexpr int kMaxDev = 64;
    static int sms[kMaxDev] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        return 152;
    }
    int v = __atomic_load_n(&sms[dev], __ATOMIC_RELAXED);
    if (v <= 0) {
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
            cudaGetLastError();
            v = 152;
        }
        __atomic_store_n(&sms[dev], v, __ATOMIC_RELAXED);
    }
    return v;
}

}  // namespace qbvh
