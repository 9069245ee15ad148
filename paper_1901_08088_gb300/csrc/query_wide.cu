// Neighbor-list traversal over 32-wide boxes (exact lists, 32 particles per
// warp in Z-order; the rope walks of the binary tree are in query.cu).
//
// The paper collapses small subtrees into leaves and names wider nodes as the
// next step (Sec. 2.3, Sec. 5).  Leaves are contiguous in Z-order, so a node
// 32 wide needs no links: box k of level 1 bounds leaves 32 k .. 32 k + 31, box
// k of level 2 bounds 32 boxes of level 1 (1024 leaves), level 3 again (32768).
// The fit writes them (build.cu).  One warp tests the 32 children of a node at
// once, one per lane, against its packet: the box of its particles' image
// centres grown by the search radius.  A walk is then a few ballots instead of
// a chain of dependent node visits (N = 2,097,152, density 0.8, radius 3.3: 127
// nodes and 26 bundles of the binary tree per packet before).
//
// A run of 32 leaves is not aligned to the cells of the Z-order: a run that
// crosses from one octant to the next holds the far corner of the first and the
// near corner of the second, and its bounding box spans both octants.  One run
// in eight crosses a cell boundary one level up, one in 64 two levels up, so
// that with one box per run every level adds the same number of false overlaps
// (N = 1,000,000, density 0.2: traversal 2.65 ms against 0.65 ms of the rope
// walk).  So every node holds two boxes, of the leaves before and after the
// highest cell boundary inside it (bit by bit the top split of the binary tree
// over its keys); either side is then compact.  A packet of particles has the
// same two sides, and keeps them apart where that covers less.
//
// Nodes are not aligned to trees: where two trees meet, one node bounds leaves
// of both, which only makes it larger; leaves outside the tree are masked.
//
// Work of one packet, per tree and periodic image:
//   1. the boxes that the packet overlaps, in Z-order, down to 32-leaf chunks;
//   2. a chunk's leaves against the packet's box, one per lane; survivors are
//      appended to a stage in shared memory;
//   3. every 32 staged survivors are tested by every lane against its own
//      particle: t = |u_j - x_i|^2 - r^2 by fused multiply-adds on packed pairs,
//      u_j = fl(x_j - nL) as staged, the sign of t shifted into a 32-bit mask (5
//      to 6 instructions per survivor).  Survivors of different images share
//      a group.  t is not the list's decision; it decides outside a band around
//      0, and a group's pairs with |t| inside the band are decided by the pinned
//      expression on the leaves.  The band, with u = 2^-24:
//      zero image: u_j = x_j, the components are the pinned ones, d2 and t differ
//      by at most 6.1 u r^2 where d2 is near r^2; band 2^-20 r^2 (16 u r^2).  Far
//      from r^2 both errors stay below 4 u d2, which cannot cross the band;
//      other images: fl(u_j - x_i) and the pinned fl(fl(x_j - x_i) - nL) differ by
//      at most 3 u L + 2 u r < e = 2^-21 L per component, so d2 and t by less than
//      8 r e + 4 e^2 + 2^-20 (r + e)^2, which is added to the band;
//   4. every kPool groups each lane writes the survivors of its masks to its
//      row through the staging ring.  Lanes accept different survivors, and a
//      warp takes as many steps as its fullest lane has entries: 214 steps for
//      119 entries a lane with pools of 7 groups at N = 262,144, about 150 with
//      14, two to three times the mean with one.
//
// Rows hold a particle's neighbours tree by tree, image by image, in Z-order --
// the order of the rope walk with one particle per lane, whatever the number of
// lanes per particle here.
//
// Conservativeness: the packet's box contains the image centre of every lane
// that walks the image, and a chunk's box contains its leaves, so the gap
// between the boxes, rounded down, never exceeds the distance that query.cu's
// header bounds by the padded radius; the test keeps every box and leaf that
// some lane's exact test could accept.
//
// Measured (whole query, rope walk before -> here, microseconds): N = 1000 181 -> 20;
// 30,011 256 -> 61; 131,072 with r = 1.42 190 -> 67; 131,072 in double precision 339
// -> 130; 262,144 327 -> 161; the L = 100 mixture 576 -> 251; liquid/vapor 1,000,000
// 646 -> 399; 32 x 65,536 1523 -> 1029; 256 uneven systems 1904 -> 1236; 2,097,152
// 1242 -> 959.  Bound by instruction issue and shared memory
// together (N = 262,144: 62% of the issue rate, 58% of the L1 data pipe); leaving
// parts out at N = 2,097,152 put 39% of the time in writing the rows, 25% in the
// group tests, 20% in the chunks' filter, 16% in boxes and set-up.  One code path
// for every image matters: with a second one for the zero image the uneven systems
// stalled on instruction fetch.
#include <stddef.h>

#include "query_common.cuh"

namespace qbvh {

namespace {

constexpr int kPool = 14;   // groups whose masks wait; a tree's last, partial group may add one

// lanes per particle W: 1 (stage, masks and row rings), 4 (stage only), 32 (none)
template <int W>
struct __align__(16) WideStage {
    float x[64], y[64], z[64];        // survivors, slot = running index & 63
    int zid[64];                      // their Z-order indices, -1 for padding
    int id[W == 1 ? 512 : 64];        // their original indices (W = 1: of the pool and the stage, from
                                      // the pool's first, reversed within a group: mask bit p
                                      // belongs to slot p)
    unsigned mask[W == 1 ? kPool + 1 : 1][32];
    int ring[W == 1 ? 16 * 32 : 4];   // slot k of lane l at ring[32 k + l]
};

template <int W>
constexpr size_t stage_size()
{
    return W == 32 ? 0 : sizeof(WideStage<W>);
}

struct OutRow {
    int *row;
    int cap;
    int count;   // accepted entries of the particle (W = 1: of the lane)
    int base;    // W = 1: entries [0, base) have left the ring (a multiple of 8)
};

// running indices of the warp's survivors, over all its walks
struct Walk {
    int tot;     // staged
    int tested;  // tested (a multiple of 32)
    int pool;    // first one whose group's masks wait in the pool
    int self;    // index of the lane's own particle among the survivors, or -1
};

__device__ __forceinline__ unsigned lanes_below()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

struct Box {
    float lx, ly, lz, hx, hy, hz;
};

// squared gap between two boxes, rounded down
__device__ __forceinline__ float gap2(const Box &a, const Box &b)
{
    const float gx = fmaxf(fmaxf(__fsub_rd(a.lx, b.hx), __fsub_rd(b.lx, a.hx)), 0.f);
    const float gy = fmaxf(fmaxf(__fsub_rd(a.ly, b.hy), __fsub_rd(b.ly, a.hy)), 0.f);
    const float gz = fmaxf(fmaxf(__fsub_rd(a.lz, b.hz), __fsub_rd(b.lz, a.hz)), 0.f);
    return __fmaf_rd(gx, gx, __fmaf_rd(gy, gy, __fmul_rd(gz, gz)));
}

// the packet's search centres: one box, or two where that covers less
struct Packet {
    Box a, b;
    bool two;   // warp-uniform
};

__device__ __forceinline__ bool near_packet(const Packet &p, const Box &n, float rs2)
{
    float g = gap2(p.a, n);
    if (p.two) g = fminf(g, gap2(p.b, n));
    return g <= rs2;
}

// children base .. base + 31 of a node, those in [first, last], against the packet
// (an empty side holds lower corners of +inf: its gap is infinite)
__device__ __forceinline__ unsigned test_boxes(const float4 *boxes, int base, int first, int last, const Packet &p,
                                               float rs2)
{
    const int i = base + (int)(threadIdx.x & 31);
    bool hit = false;
    if (i >= first && i <= last) {
        float4 a, b, c, d;
        node32_ld(boxes + 4 * (size_t)i, a, b);
        node32_ld(boxes + 4 * (size_t)i + 2, c, d);
        hit = near_packet(p, Box{a.x, a.y, a.z, a.w, b.x, b.y}, rs2) ||
              near_packet(p, Box{c.x, c.y, c.z, c.w, d.x, d.y}, rs2);
    }
    return __ballot_sync(FULL, hit);
}

// Box of the image centres fl(x_i + n L) of the lanes in `on`.  Positions are in
// [0, L): their bit patterns order like the values once -0 is folded into +0,
// and fl(x + n L) is monotone in x.
__device__ __forceinline__ Box centre_box(const Query &c, bool on)
{
    const unsigned bx = __float_as_uint(c.xi + 0.f), by = __float_as_uint(c.yi + 0.f), bz = __float_as_uint(c.zi + 0.f);
    Box p;
    p.lx = __fadd_rn(__uint_as_float(__reduce_min_sync(FULL, on ? bx : 0x7F800000u)), c.nLx);
    p.ly = __fadd_rn(__uint_as_float(__reduce_min_sync(FULL, on ? by : 0x7F800000u)), c.nLy);
    p.lz = __fadd_rn(__uint_as_float(__reduce_min_sync(FULL, on ? bz : 0x7F800000u)), c.nLz);
    p.hx = __fadd_rn(__uint_as_float(__reduce_max_sync(FULL, on ? bx : 0u)), c.nLx);
    p.hy = __fadd_rn(__uint_as_float(__reduce_max_sync(FULL, on ? by : 0u)), c.nLy);
    p.hz = __fadd_rn(__uint_as_float(__reduce_max_sync(FULL, on ? bz : 0u)), c.nLz);
    return p;
}

__device__ __forceinline__ float grown_volume(const Box &b, float d)
{
    return (b.hx - b.lx + d) * (b.hy - b.ly + d) * (b.hz - b.lz + d);
}

// the lanes in `on`, those of each side of the packet's split apart
__device__ __forceinline__ Packet make_packet(const Query &c, bool on, bool side, float rs)
{
    Packet p;
    p.a = centre_box(c, on && !side);
    p.two = false;
    const unsigned left = __ballot_sync(FULL, on && !side), right = __ballot_sync(FULL, on && side);
    if (right == 0u) return p;
    p.b = centre_box(c, on && side);
    if (left == 0u) {
        p.a = p.b;
        return p;
    }
    const Box u{fminf(p.a.lx, p.b.lx), fminf(p.a.ly, p.b.ly), fminf(p.a.lz, p.b.lz),
                fmaxf(p.a.hx, p.b.hx), fmaxf(p.a.hy, p.b.hy), fmaxf(p.a.hz, p.b.hz)};
    const float d = 2.f * rs;
    p.two = grown_volume(p.a, d) + grown_volume(p.b, d) < 0.95f * grown_volume(u, d);
    if (!p.two) p.a = u;
    return p;
}

// The list's decision for leaf j (position q) under the image in c.
template <bool F64>
__device__ __forceinline__ bool decide(const QueryArgs &a, const Query &c, int j, const float4 &q)
{
    const float d2 = exact_d2<true>(c, q);
    if (!F64) return d2 < c.rl2;
    if (d2 < c.rl2_lo) return true;
    return d2 <= c.rl2_hi && exact_d2_64<true>(a, c, j) < a.r2_64[c.pair];
}

// Mask of the 32 survivors starting at slot s0 against the lane's particle,
// first survivor in bit 31.  With W = 4 the lane tests survivors 8 wsub ..
// 8 wsub + 7 and the group's lanes combine.  Every lane of the warp calls this
// together.
template <bool F64, int W>
__device__ __forceinline__ unsigned group_mask(const QueryArgs &a, const Query &c, const WideStage<W> *st, int s0,
                                               int wsub, float band, float L)
{
    constexpr int N = 32 / W;
    const int o = s0 + N * wsub;
    const f32x2 xi = f2_pack(c.xi, c.xi), yi = f2_pack(c.yi, c.yi), zi = f2_pack(c.zi, c.zi);
    const f32x2 r2 = f2_pack(-c.rl2, -c.rl2);
    unsigned m = 0u;
    float near = __int_as_float(0x7F800000);
#pragma unroll
    for (int k = 0; k < N; k += 4) {
        const float4 X = *reinterpret_cast<const float4 *>(st->x + o + k);
        const float4 Y = *reinterpret_cast<const float4 *>(st->y + o + k);
        const float4 Z = *reinterpret_cast<const float4 *>(st->z + o + k);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const f32x2 dx = f2_sub(h ? f2_pack(X.z, X.w) : f2_pack(X.x, X.y), xi);
            const f32x2 dy = f2_sub(h ? f2_pack(Y.z, Y.w) : f2_pack(Y.x, Y.y), yi);
            const f32x2 dz = f2_sub(h ? f2_pack(Z.z, Z.w) : f2_pack(Z.x, Z.y), zi);
            float t0, t1;
            f2_unpack(f2_fma(dx, dx, f2_fma(dy, dy, f2_fma(dz, dz, r2))), t0, t1);
            m = __funnelshift_l(__float_as_uint(t0), m, 1);
            m = __funnelshift_l(__float_as_uint(t1), m, 1);
            near = fminf(fminf(near, fabsf(t0)), fabsf(t1));
        }
    }
    if (__any_sync(FULL, !(near > band))) {
        // some pair lies in the band: the pinned expression decides it, the image
        // being the whole multiple of L between leaf and staged point
#pragma unroll 1
        for (int k = 0; k < N; ++k) {
            const float ux = st->x[o + k], uy = st->y[o + k], uz = st->z[o + k];
            const float dx = __fsub_rn(ux, c.xi), dy = __fsub_rn(uy, c.yi), dz = __fsub_rn(uz, c.zi);
            const float t = __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmaf_rn(dz, dz, -c.rl2)));
            const int j = st->zid[o + k];
            if (!(fabsf(t) > band) && j >= 0) {
                const float4 q = tree_ld(a.leaves + j);
                Query e = c;
                e.nLx = L * rintf((q.x - ux) / L);
                e.nLy = L * rintf((q.y - uy) / L);
                e.nLz = L * rintf((q.z - uz) / L);
                const unsigned bit = 1u << (N - 1 - k);
                m = decide<F64>(a, e, j, q) ? m | bit : m & ~bit;
            }
        }
    }
    if (W > 1) {
        m <<= 32 - N - N * wsub;
#pragma unroll
        for (int k = 16; k >= 32 / W; k >>= 1) m |= __shfl_xor_sync(FULL, m, k);
    }
    return m;
}

// One step of emit_pool: the highest set bit p of the lane's mask m takes its
// survivor's index from the group's slots (group base g) to the ring at byte
// offset off; an empty mask gives way to the next group's.  Without a set bit the
// store goes to the free slot after the last entry (the load, four bytes before
// the group's first slot, stays inside the stage).  Written out so that nothing
// here is a branch: 15 instructions, where the compiled conditions took about 33
// (N = 2,097,152: 1013 -> 953 us, 80 registers both).  What is left of it is shared
// memory: 32 lanes read 32 places of the pool's indices, three to four
// wavefronts.
__device__ __forceinline__ void emit_step(unsigned &m, unsigned &off, unsigned &g, unsigned last, unsigned ring,
                                          unsigned lane4)
{
    asm volatile(
        "{\n"
        ".reg .pred some, left, next;\n"
        ".reg .u32 p, t, id;\n"
        "bfind.u32 p, %0;\n"
        "setp.ne.u32 some, %0, 0;\n"
        "shl.b32 t, p, 2;\n"
        "add.u32 t, t, %2;\n"
        "ld.shared.u32 id, [t + %6];\n"
        "add.u32 t, %4, %1;\n"
        "st.shared.u32 [t], id;\n"
        "@some add.u32 %1, %1, 128;\n"
        "and.b32 %1, %1, 0x780;\n"
        "shl.b32 t, 1, p;\n"          // 0 for an empty mask: p = -1 is clamped
        "not.b32 t, t;\n"
        "and.b32 %0, %0, t;\n"
        "setp.ne.u32 left, %2, %3;\n"
        "setp.eq.and.u32 next, %0, 0, left;\n"
        "@next add.u32 %2, %2, 128;\n"
        "@next add.u32 t, %2, %5;\n"
        "@next ld.shared.u32 %0, [t + %7];\n"
        "}\n"
        : "+r"(m), "+r"(off), "+r"(g)
        : "r"(last), "r"(ring), "r"(lane4), "n"(offsetof(WideStage<1>, id)), "n"(offsetof(WideStage<1>, mask))
        : "memory");
}

// W = 1: the pool's survivors to the lanes' rows, each lane its own masks in
// order, one entry per step; completed sectors leave the ring once per 8 steps
// (at most 15 entries wait in its 16 slots).  A step either takes a bit or moves
// to the next mask, so the loop ends.
__device__ __forceinline__ void emit_pool(WideStage<1> *st, OutRow &out, Walk &w)
{
    const int lane = threadIdx.x & 31;
    const int groups = (w.tested - w.pool) >> 5;
    const unsigned base = (unsigned)__cvta_generic_to_shared(st);
    const unsigned ring = (unsigned)__cvta_generic_to_shared(st->ring + lane);
    unsigned off = (out.count & 15) << 7;    // byte offset of the next free slot
    unsigned boff = (out.base & 15) << 7;    // and of the first entry
    unsigned g = base;
    const unsigned last = base + 128 * (groups - 1);
    unsigned m = st->mask[0][lane];
    do {
#pragma unroll
        for (int u = 0; u < 8; ++u) emit_step(m, off, g, last, ring, 4 * lane);
        if (((off - boff) & 0x780) >= 8 * 128) {
            if (out.base + 8 <= out.cap) store_sector(out.row + out.base, st->ring + lane + (boff >> 2));
            out.base += 8;
            boff ^= 8 * 128;
        }
    } while (__any_sync(FULL, m != 0u || g != last));
    out.count = out.base + (((off - boff) & 0x780) >> 7);
    // the staged survivors that wait for their group come first in the next pool
    const int rest = st->id[32 * groups + lane];
    __syncwarp();
    st->id[lane] = rest;
    w.pool = w.tested;
    __syncwarp();
}

// one group of 32 staged survivors
template <bool F64, int W>
__device__ __forceinline__ void take_group(const QueryArgs &a, const Query &c, OutRow &out, WideStage<W> *st, Walk &w,
                                           bool part, int wsub, float band, float L)
{
    __syncwarp();   // the group's survivors are staged
    const int s0 = w.tested & 63;
    unsigned m = group_mask<F64, W>(a, c, st, s0, wsub, band, L);
    if ((w.self >> 5) == (w.tested >> 5)) m &= ~(0x80000000u >> (w.self & 31));
    if (!part) m = 0u;
    if (W == 1) {
        st->mask[(w.tested - w.pool) >> 5][threadIdx.x & 31] = m;
    } else {
        constexpr int N = 32 / W;
        unsigned mine = (m << (N * wsub)) & ~(0xFFFFFFFFu >> N);
        int pos = out.count + __popc(m & ~(0xFFFFFFFFu >> (N * wsub)));
        const int *ids = st->id + s0 + N * wsub;
        while (mine) {
            const int b = __clz((int)mine);
            if (pos < out.cap) row_store(out.row + pos, ids[b]);
            ++pos;
            mine &= 0x7FFFFFFFu >> b;
        }
        out.count += __popc(m);
    }
    w.tested += 32;
    __syncwarp();   // and read: their slots may be reused
}

// The packet's walk of the tree holding leaves [first, last] under one image.
// on: lanes whose sphere reaches the tree under the image.  part: lanes whose
// particles walk this tree.  side: the lane's side of the packet's split.  own:
// the chunk holding the packet's own particles under the zero image, or -1;
// own_lane: the lane whose leaf of that chunk is this lane's particle.
template <bool F64, int W>
__device__ __forceinline__ void wide_walk(const QueryArgs &a, const Query &c, OutRow &out, WideStage<W> *st, Walk &w,
                                          int first, int last, bool on, bool part, bool side, float rs, float rs2,
                                          float band, float L, int own, int own_lane, int wsub)
{
    const int lane = threadIdx.x & 31;
    Packet p;
    if (W == 32) {
        p.a = Box{c.px, c.py, c.pz, c.px, c.py, c.pz};
        p.two = false;
    } else {
        p = make_packet(c, on, side, rs);
    }
    const int a3 = first >> 15, b3 = last >> 15;
    for (int n3 = a3; n3 <= b3; n3 += 32) {
        // a level with one node in the tree's range is not tested
        unsigned M3 = a3 == b3 ? 1u : test_boxes(a.box3, n3, a3, b3, p, rs2);
        while (M3) {
            const int c3 = (n3 + __ffs(M3) - 1) << 5;
            M3 &= M3 - 1u;
            const int a2 = max(first >> 10, c3), b2 = min(last >> 10, c3 + 31);
            unsigned M2 = a2 == b2 ? 1u << (a2 & 31) : test_boxes(a.box2, c3, a2, b2, p, rs2);
            while (M2) {
                const int c2 = (c3 + __ffs(M2) - 1) << 5;
                M2 &= M2 - 1u;
                unsigned M1 = test_boxes(a.box1, c2, first >> 5, last >> 5, p, rs2);
                // the next chunk's leaves are loaded while this one's are tested
                float4 qn = make_float4(0.f, 0.f, 0.f, 0.f);
                if (M1) qn = tree_ld(a.leaves + min(((c2 + __ffs(M1) - 1) << 5) + lane, last));
                while (M1) {
                    const int chunk = c2 + __ffs(M1) - 1;
                    M1 &= M1 - 1u;
                    const float4 q = qn;
                    if (M1) qn = tree_ld(a.leaves + min(((c2 + __ffs(M1) - 1) << 5) + lane, last));
                    const int j = (chunk << 5) + lane;
                    const bool in = j >= first && j <= last;
                    const int id = __float_as_int(q.w) & 0x7FFFFFFF;
                    if (W == 32) {
                        const bool acc = in && j != c.self && decide<F64>(a, c, j, q);
                        const unsigned m = __ballot_sync(FULL, acc);
                        if (acc) {
                            const int pos = out.count + __popc(m & lanes_below());
                            if (pos < out.cap) row_store(out.row + pos, id);
                        }
                        out.count += __popc(m);
                        continue;
                    }
                    if (W == 1 && w.tested - w.pool >= 32 * kPool) emit_pool(reinterpret_cast<WideStage<1> *>(st), out, w);
                    const bool surv = in && near_packet(p, Box{q.x, q.y, q.z, q.x, q.y, q.z}, rs2);
                    const unsigned S = __ballot_sync(FULL, surv);
                    const int r = w.tot + __popc(S & lanes_below());
                    if (surv) {
                        const int k = r & 63;
                        st->x[k] = __fsub_rn(q.x, c.nLx);
                        st->y[k] = __fsub_rn(q.y, c.nLy);
                        st->z[k] = __fsub_rn(q.z, c.nLz);
                        st->zid[k] = j;
                        st->id[W == 1 ? (r - w.pool) ^ 31 : k] = id;
                    }
                    // the packet's own chunk hands every lane its own particle
                    // (a survivor wherever the lane walks this tree as its own)
                    if (chunk == own) {
                        const int ro = __shfl_sync(FULL, surv ? r : -1, own_lane);
                        w.self = part ? ro : -1;
                    }
                    w.tot += __popc(S);
                    if (w.tot - w.tested >= 32) take_group<F64, W>(a, c, out, st, w, part, wsub, band, L);
                }
            }
        }
    }
}

// every tree of system `sys` under every image, for the particles (type ta) of
// the lanes in `part`
template <bool F64, int W>
__device__ __forceinline__ void walk_trees(const QueryArgs &a, Query &c, OutRow &out, WideStage<W> *st, Walk &w, int sys,
                                           int ta, int T, bool part, bool side, int own, int own_lane, int wsub)
{
    const int lane = threadIdx.x & 31;
    const float L = a.sys[sys].L;
    for (int tb = 0; tb < T; ++tb) {
        const int pair = ta * T + tb;
        const float r = a.r_list[pair];
        if (!(r > 0.f)) continue;
        const SegInfo &g = a.seg[sys * T + tb];
        const int first = g.start, last = g.start + g.count - 1;
        if (last < first) continue;
        const float rs2 = a.rs2[pair];
        c.rl2 = a.rl2[pair];
        if (F64) {
            c.rl2_lo = a.rl2_lo[pair];
            c.rl2_hi = a.rl2_hi[pair];
            c.pair = pair;
        }
        // most packets see the tree under the zero image alone: no shift by L brings
        // a lane's sphere to the root box on any axis (the rounding here, below
        // 2^-22 L, is inside the 2^-19 L that rs adds to the radius)
        const float rs = a.rs[pair];
        const bool inner = c.xi - L + rs < g.rlo[0] && c.xi + L - rs > g.rhi[0] && c.yi - L + rs < g.rlo[1] &&
                           c.yi + L - rs > g.rhi[1] && c.zi - L + rs < g.rlo[2] && c.zi + L - rs > g.rhi[2];
        unsigned mine = part ? 1u << 13 : 0u;
        if (!__all_sync(FULL, inner || !part)) mine = part ? image_mask(c.xi, c.yi, c.zi, L, g, rs2) : 0u;
        unsigned mask = __reduce_or_sync(FULL, mine);
        // band of the group test (header comment); every group is decided by the
        // pinned expression where r^2 is too small or too large for the bounds
        float band = c.rl2 * 9.5367431640625e-7f;
        if (F64) band += fmaxf(c.rl2_hi - c.rl2, c.rl2 - c.rl2_lo);
        if (mask & ~(1u << 13)) {
            const float e = L * 4.76837158203125e-7f;
            band += 8.f * r * e + 4.f * e * e + (r + e) * (r + e) * 9.5367431640625e-7f;
        }
        if (!(c.rl2 > 1e-30f && c.rl2 < 1e30f)) band = __int_as_float(0x7F800000);
        while (mask) {
            const int img = __ffs(mask) - 1;
            mask &= mask - 1u;
            set_image(c, img, L);
            wide_walk<F64, W>(a, c, out, st, w, first, last, (mine >> img) & 1u, part, side, rs, rs2, band, L,
                              img == 13 && tb == ta ? own : -1, own_lane, wsub);
        }
        if (W < 32 && w.tot > w.tested) {
            // the tree's last group, padded with points that no lane accepts
            // (their squared distance overflows to +inf)
            if (lane >= w.tot - w.tested) {
                const int s = (w.tested + lane) & 63;
                st->x[s] = st->y[s] = st->z[s] = 1e30f;
                st->zid[s] = -1;
            }
            w.tot = w.tested + 32;
            take_group<F64, W>(a, c, out, st, w, part, wsub, band, L);
        }
    }
}

__device__ __forceinline__ int row_index(const QueryArgs &a, int s, const float4 &me)
{
    const int i = __float_as_int(me.w) & 0x7FFFFFFF;
    if (i < a.n) return i;
    atomicOr(&a.status->err, QBVH_DEVERR_INTERNAL);
    return s;
}

// one particle by the whole warp (W = 32)
template <bool F64>
__device__ __forceinline__ int walk_particle(const QueryArgs &a, int s, int seg, int T)
{
    const float4 me = __ldg(a.leaves + s);
    const int i = row_index(a, s, me);
    Query c;
    c.xi = me.x;
    c.yi = me.y;
    c.zi = me.z;
    c.self = s;
    OutRow out{a.rows + (size_t)i * a.cap, a.cap, 0, 0};
    Walk w{0, 0, 0, -1};
    const int sys = seg / T;
    walk_trees<F64, 32>(a, c, out, nullptr, w, sys, seg - sys * T, T, true, false, -1, 0, 0);
    if ((threadIdx.x & 31) == 0) a.counts[i] = out.count;
    return out.count;
}

// the leading blocks: every particle of a sparse tree (query_common.cuh) gets a warp
__device__ __forceinline__ void sparse_walks(const QueryArgs &a)
{
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)((a.sparse_blocks * blockDim.x) >> 5);
    for (int ta = 0; ta < a.n_types; ++ta) {
        if (!sparse_tree(a, ta)) continue;
        const int start = a.seg[ta].start, count = a.seg[ta].count;
        for (int p = gw; p < count; p += nw) warp_max_count(walk_particle<false>(a, start + p, ta, a.n_types), a.status);
    }
}

// ---- spread packets --------------------------------------------------------
// The boxes around far-apart particles (a dilute type among a dense one, vapor around
// a droplet) cover most of the system, and the packet's warp would test most of its
// leaves, alone and long after the others.  Spread is a run of 32 leaves that holds
// particles whose boxes, grown by the radius, cover more than kSpreadVolume times
// what the cubes around 32 separate spheres do and reach more than kSpreadChunks
// chunks of leaves under the zero image: a gas stays with its packets, which find
// little.  spread_kernel marks these runs and walks their particles one per warp; the
// packets' walk passes over them.  The rows are the same either way.
//
// Query, milliseconds, walk of the binary tree / packets alone / this: 64 particles of
// a second type among 2,000,000 in double precision 5.1 / 28.9 / 1.9; four types of 64
// among 2,000,000 of a fifth 4.1 / 27.2 / 1.7; four batched systems of 250,000 with 32
// each 3.3 / 5.9 / 0.85; a droplet of 1,000,000 with 100,000 vapor particles in a box
// of 4000, radius 1.2, 1.07 / 1.61 / 0.34; 31 particles listed only against 1,000,000 of
// another type in double precision 3.0 / 20.3 / 0.11.  It costs 2 to 4 us per query (N = 30,011 58 ->
// 61, 131,072 with r = 1.42 65 -> 67, 2,097,152 953 -> 959), and a gas of 1,000,000 at
// density 0.0005 the counting of its chunks, 119 -> 167 us (binary tree 224).
//
// Four times: up to there a packet tests at most about 30,000 leaves at density 0.8
// and radius 3.3, fewer than the walk of the binary tree did (44,000).  128 chunks are
// four per particle: a particle by itself visits 20 to 25 there.
constexpr float kSpreadVolume = 4.f;
constexpr int kSpreadChunks = 128;
constexpr int kSpreadRuns = 8;   // most runs per warp of spread_kernel

__device__ __forceinline__ int chunks_reached(const QueryArgs &a, int first, int last, const Packet &p, float rs2, int n)
{
    for (int n3 = first >> 15; n3 <= last >> 15; n3 += 32) {
        unsigned M3 = test_boxes(a.box3, n3, first >> 15, last >> 15, p, rs2);
        while (M3) {
            const int c3 = (n3 + __ffs(M3) - 1) << 5;
            M3 &= M3 - 1u;
            unsigned M2 = test_boxes(a.box2, c3, first >> 10, last >> 10, p, rs2);
            while (M2) {
                n += __popc(test_boxes(a.box1, (c3 + __ffs(M2) - 1) << 5, first >> 5, last >> 5, p, rs2));
                if (n > kSpreadChunks) return n;
                M2 &= M2 - 1u;
            }
        }
    }
    return n;
}

__device__ __forceinline__ int seg_of_leaf(const QueryArgs &a, int s)
{
    return a.wide_keys ? seg_of_sorted<true>(a, s) : seg_of_sorted<false>(a, s);
}

__device__ __forceinline__ unsigned code_of_leaf(const QueryArgs &a, int s)   // 30-bit Z-order code
{
    return QBVH_QMASK & (a.wide_keys ? (unsigned)__ldg(reinterpret_cast<const unsigned long long *>(a.keys_sorted) + s)
                                     : __ldg(reinterpret_cast<const unsigned *>(a.keys_sorted) + s));
}

// The side of the highest cell boundary inside the particles of the lanes in `part`:
// the top bit in which their first and last codes differ.
__device__ __forceinline__ bool split_side_of(unsigned code, bool part)
{
    const unsigned who = __ballot_sync(FULL, part);
    const unsigned x = __shfl_sync(FULL, code, __ffs(who) - 1) ^ __shfl_sync(FULL, code, 31 - __clz((int)who));
    return x != 0u && ((code >> (31 - __clz((int)x))) & 1u);
}

__device__ __forceinline__ bool spread_volume(const Box &a, const Box &b, bool two, float rs)
{
    const float d = 2.f * rs;
    return grown_volume(a, d) + (two ? grown_volume(b, d) : 0.f) > kSpreadVolume * 32.f * d * d * d;
}

// Comes before the packets' walk.  A block takes every gridDim.x-th run, `runs` per
// warp (spread ones lie side by side), and shares the particles of the spread ones it
// finds among its warps.  A lane compares its run's volume with the smallest sphere
// of the list; for the runs that this leaves, the warp tries every tree that has
// particles in the run, with those particles' boxes and that tree's radii (a few
// particles of a dilute type may follow the last ones of a type that has no list of
// its own).
template <bool F64>
__global__ void __launch_bounds__(256, 4) spread_kernel(const __grid_constant__ QueryArgs a, int runs)
{
    __shared__ int s_run[8 * kSpreadRuns];
    __shared__ int s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, T = a.n_types;
    const long long run = ((threadIdx.x >> 5) * runs + lane) * (long long)gridDim.x + blockIdx.x;
    bool wide = false;
    if (lane < runs && 32 * run < a.n) {
        float rs = __int_as_float(0x7F800000);
        for (int k = 0; k < T * T; ++k)
            if (a.r_list[k] > 0.f) rs = fminf(rs, a.rs[k]);
        float4 b[4];
        node32_ld(a.box1 + 4 * run, b[0], b[1]);
        node32_ld(a.box1 + 4 * run + 2, b[2], b[3]);
        // (an empty side has lower corners of +inf)
        wide = spread_volume(Box{b[0].x, b[0].y, b[0].z, b[0].w, b[1].x, b[1].y},
                             Box{b[2].x, b[2].y, b[2].z, b[2].w, b[3].x, b[3].y}, b[2].x <= b[2].w, rs);
    }
    bool mark = false;
    unsigned todo = __ballot_sync(FULL, wide);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int s = 32 * (int)__shfl_sync(FULL, run, src) + lane;
        const int seg = s < a.n ? seg_of_leaf(a, s) : -1;
        const unsigned code = s < a.n ? code_of_leaf(a, s) : 0u;
        const float4 me = __ldg(a.leaves + min(s, a.n - 1));
        Query c{};
        c.xi = me.x;
        c.yi = me.y;
        c.zi = me.z;
        bool found = false;
        unsigned rest = __ballot_sync(FULL, seg >= 0);
        while (rest && !found) {
            const int sg = __shfl_sync(FULL, seg, __ffs(rest) - 1), sys = sg / T, ta = sg - sys * T;
            const bool part = seg == sg;
            rest &= ~__ballot_sync(FULL, part);
            // (a sparse tree has its own walk)
            if (!F64 && a.sparse_blocks > 0 && sparse_tree(a, sg)) continue;
            int n = 0;
            for (int tb = 0; tb < T && n <= kSpreadChunks; ++tb) {
                const SegInfo &g = a.seg[sys * T + tb];
                const float rs = a.rs[ta * T + tb];
                if (!(a.r_list[ta * T + tb] > 0.f) || g.count == 0) continue;
                const Packet q = make_packet(c, part, split_side_of(code, part), rs);
                if (spread_volume(q.a, q.b, q.two, rs))
                    n = chunks_reached(a, g.start, g.start + g.count - 1, q, a.rs2[ta * T + tb], n);
            }
            found = n > kSpreadChunks;
        }
        if (lane == src) mark = found;
    }
    if (lane < runs && 32 * run < a.n) {
        a.spread[run] = mark;
        if (mark) s_run[atomicAdd(&s_n, 1)] = (int)run;
    }
    __syncthreads();
    // (at the start, the walk's blocks would be placed around this kernel's: N = 30,011
    // 72 us instead of 62)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int k = threadIdx.x >> 5; k < 32 * s_n; k += 8) {
        const int s = 32 * s_run[k >> 5] + (k & 31);
        if (s >= a.n) continue;
        const int sg = seg_of_leaf(a, s);
        if (!F64 && a.sparse_blocks > 0 && sparse_tree(a, sg)) continue;
        warp_max_count(walk_particle<F64>(a, s, sg, T), a.status);
    }
}

// ONE: a single tree (one system, one type).  Registers: 80 (24 warps per SM) for
// one particle per lane, which spills under 64 (32 warps): N = 2,097,152 1039 -> 953
// us, liquid/vapor 1,000,000 434 -> 393, the L = 100 mixture 290 -> 248; 48 registers
// (40 warps) were slower still.  A single tree of double-precision data, whose FP64
// decision is rare, is 133 us with 64 and 139 with 80 (N = 131,072).
template <bool ONE, bool F64, int W>
__global__ void __launch_bounds__(256, W == 1 && !(ONE && F64) ? 3 : 4) wide_query_kernel(const __grid_constant__ QueryArgs a)
{
    constexpr int G = 32 / W;
    // (double-precision data: waiting here took 8 us more than a plain launch, N = 131,072)
    if (W < 32 && !F64) pdl_begin();
    int blk = (int)blockIdx.x, nblk = (int)gridDim.x;
    const bool sparse = !ONE && !F64 && a.sparse_blocks > 0;
    if (sparse) {
        if (blk < a.sparse_blocks) {
            sparse_walks(a);
            return;
        }
        blk -= a.sparse_blocks;
        nblk -= a.sparse_blocks;
    }
    const int T = ONE ? 1 : a.n_types;
    // several types: the last trees first (query_common.cuh, sparse trees)
    if (!ONE && T > 1) blk = nblk - 1 - blk;
    const int packet = (int)((blk * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    const int pidx = lane % G, wsub = lane / G;
    const int s = packet * G + pidx;
    const bool active = s < a.n;
    const int seg_i = !active ? -1 : (ONE ? 0 : (a.wide_keys ? seg_of_sorted<true>(a, s) : seg_of_sorted<false>(a, s)));
    if (W == 32) {
        if (!active || (sparse && sparse_tree(a, seg_i))) return;
        warp_max_count(walk_particle<F64>(a, s, seg_i, T), a.status);
        return;
    }
    // walked by spread_kernel (a single tree leaves here, others pass over their trees:
    // one return too many cost 32 x 65,536 particles 6 us, one flag too many 8 at 2,097,152)
    const bool marked = packet * G < a.n && __ldcg(a.spread + ((packet * G) >> 5)) != 0;
    if (ONE && marked) return;
    const float4 me = active ? __ldg(a.leaves + s) : make_float4(0.f, 0.f, 0.f, 0.f);
    const int i = active ? row_index(a, s, me) : 0;
    const unsigned code = active ? code_of_leaf(a, s) : 0u;
    Query c;
    c.xi = me.x;
    c.yi = me.y;
    c.zi = me.z;
    c.self = active ? s : 0;   // an idle lane's tests read a valid particle too
    OutRow out{a.rows + (size_t)i * a.cap, a.cap, 0, 0};
    Walk w{0, 0, 0, -1};
    extern __shared__ __align__(16) unsigned char smem[];
    WideStage<W> *st = reinterpret_cast<WideStage<W> *>(smem) + (threadIdx.x >> 5);
    bool elsewhere = !ONE && marked;   // or particle of a sparse tree: walked by the leading blocks
    // the warp's particles may belong to several trees: one tree at a time
    unsigned remaining = __ballot_sync(FULL, active && !elsewhere);
    while (remaining) {
        const int seg = ONE ? 0 : __shfl_sync(FULL, seg_i, __ffs(remaining) - 1);
        const bool part = ONE ? active : (active && seg_i == seg);
        remaining = ONE ? 0u : (remaining & ~__ballot_sync(FULL, part));
        if (sparse && sparse_tree(a, seg)) {
            elsewhere = elsewhere || part;
            continue;
        }
        const int sys = ONE ? 0 : seg / T;
        const bool side = split_side_of(code, part);
        walk_trees<F64, W>(a, c, out, st, w, sys, ONE ? 0 : seg - sys * T, T, part, side, (packet * G) >> 5, s & 31,
                           wsub);
    }
    if (W == 1) {
        if (w.tested > w.pool) emit_pool(reinterpret_cast<WideStage<1> *>(st), out, w);
        // the last, partial sectors
        const int end = active && !elsewhere ? min(out.count, out.cap) : 0;
        for (int k = out.base; k < end; ++k) row_store(out.row + k, st->ring[32 * (k & 15) + lane]);
    }
    if (active && wsub == 0 && !elsewhere) a.counts[i] = out.count;
    warp_max_count(active && !elsewhere ? out.count : 0, a.status);
}

template <bool ONE, bool F64, int W>
void launch_w(const QueryArgs &a, int extra, cudaStream_t s)
{
    const int warps = a.block / 32;
    const int packets = (a.n + 32 / W - 1) / (32 / W);
    const int grid = (packets + warps - 1) / warps + extra;
    const size_t smem = warps * stage_size<W>();
    // blocks of 224 and 256 threads exceed the 48 KB that need no opt-in
    if (smem > 48 * 1024) allow_smem<wide_query_kernel<ONE, F64, W>>(8 * stage_size<W>());
    if (W == 32) {
        wide_query_kernel<ONE, F64, W><<<grid, a.block, smem, s>>>(a);
        return;
    }
    // few runs per warp while the grid is one wave: a gas counts them one after another
    const int total = (a.n + 31) / 32;
    int runs = 1;
    while (runs < kSpreadRuns && total > 8 * runs * 608) runs *= 2;
    spread_kernel<F64><<<(total + 8 * runs - 1) / (8 * runs), 256, 0, s>>>(a, runs);
    if (F64) wide_query_kernel<ONE, F64, W><<<grid, a.block, smem, s>>>(a);
    else launch_pdl(wide_query_kernel<ONE, F64, W>, grid, a.block, smem, s, a);
}

template <bool F64>
void launch_lanes(const QueryArgs &a, int lanes, int extra, cudaStream_t s)
{
    const bool one = !a.wide_keys && a.n_types == 1;
    if (lanes == 1) {
        if (one) launch_w<true, F64, 1>(a, extra, s);
        else launch_w<false, F64, 1>(a, extra, s);
    } else if (lanes == 4) {
        if (one) launch_w<true, F64, 4>(a, extra, s);
        else launch_w<false, F64, 4>(a, extra, s);
    } else {
        if (one) launch_w<true, F64, 32>(a, extra, s);
        else launch_w<false, F64, 32>(a, extra, s);
    }
}

}  // namespace

// Lanes per particle by the number of particles.  Few particles leave most of
// the GPU idle with 32 of them per warp, and a packet's walk is a serial chain:
// with 4 lanes per particle a warp has 8 particles, with 32 one.  Measured, whole
// query with its launches (microseconds, 32 / 4 / 1 lanes), density 0.8, radius 3.3: N =
// 4096 35 / 54 / 64; 8000 46 / 66 / 89; 14,503 58 / 68 / 80; 30,011 83 / 82 / 90; 45,000
// 111 / 110 / 98; 60,000 137 / 123 / 107.  Radius 1.42: 14,503 37 / 44 / 55; 30,011 49 /
// 47 / 54; 45,000 63 / 60 / 59; 60,000 81 / 66 / 62; 131,072 135 / 92 / 78.  (Both
// lines lie on the sides where these figures cross over: 30,000 and 40,000 would be
// closer, by up to 20 us at 8000 to 14,503 and 15 at 45,000 to 60,000.)
static int wide_lanes(int n)
{
    return n < 8000 ? 32 : (n < 60000 ? 4 : 1);
}

void launch_query_wide(QueryArgs a, cudaStream_t s)
{
    if (a.n == 0) return;
    a.sparse_blocks = 0;
    if (QBVH_SPARSE_TREES && !a.wide_keys && !a.f64 && a.n_types > 1)
        a.sparse_blocks = sm_count_current() * (256 / a.block);
    if (a.f64) launch_lanes<true>(a, wide_lanes(a.n), 0, s);
    else launch_lanes<false>(a, wide_lanes(a.n), a.sparse_blocks, s);
}

}  // namespace qbvh
