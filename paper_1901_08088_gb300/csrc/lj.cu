// Truncated-and-shifted Lennard-Jones energy over a neighbor list (Eq. 1 of
// the paper, shifted to zero at r_c as described in Sec. 1), in one fused pass
// that also produces the forces and the gradients with respect to the
// per-type-pair parameters:
//
//   s = (sig / r)^6,  s_c = (sig / r_c)^6
//   u(r)          = 4 eps (s^2 - s) - 4 eps (s_c^2 - s_c)           (r < r_c)
//   e_i           = 1/2 sum_{j in N(i)} u(r_ij)          (full list: each pair twice)
//   F_i           = sum_j 24 eps (2 s^2 - s) / r^2 (x_i - x_j)
//   dU/deps[a][b] = 1/2 sum_{i:a, j:b} u / eps
//   dU/dsig[a][b] = 1/2 sum_{i:a, j:b} (24 eps / sig) [(2 s^2 - s) - (2 s_c^2 - s_c)]
//
// Per-particle sums are FP32 in registers.  Each block covers particles of a
// single system and reduces its FP32 contributions in FP64 into one partial
// record; a second kernel adds the records of each system in a fixed order,
// so the FP64 totals are deterministic.
#include "qbvh_internal.cuh"

namespace qbvh {

namespace {

constexpr int kLJBlock = 128;

// Measured before -> here (forward and FP64 sums, microseconds): N = 30,011 97 ->
// 33; 131,072 with r = 1.12 40 -> 27; 262,144 124 -> 100; the L = 100 mixture 324 ->
// 141; liquid/vapor 1,000,000 255 -> 226; two-type gradients 32 x 65,536 773 -> 555;
// 256 uneven systems 477 -> 426; 2,097,152 646 -> 599.
//
// Register cap: 7 blocks of 128 threads.  One type, N = 2,097,152, 10 / 9 / 8 / 7
// blocks: 711 / 618 / 599 / 597 us; two types with gradients, 32 x 65,536, 9 / 8 / 7
// blocks / no cap: 580 / 568 / 551 / 683 us (lanes' gradient sums in FP32 then).
#ifndef QBVH_LJ_MIN_BLOCKS
#define QBVH_LJ_MIN_BLOCKS 7
#endif

// One chunk of a lane's row: 4 entries, -1 past the row's end.  SPREAD: the 8
// lanes of a particle take consecutive entries (lane r: k + r, k + 8 + r, ...);
// else each lane takes 4 consecutive ones in one load (rows are 16-byte aligned:
// the capacity is a multiple of 4).
template <bool SPREAD>
__device__ __forceinline__ int4 row_chunk(const int *row, int k, int sub, int c)
{
    int4 v = make_int4(-1, -1, -1, -1);
    if (SPREAD) {
        const int e = k + sub;
        if (e < c) v.x = __ldg(row + e);
        if (e + 8 < c) v.y = __ldg(row + e + 8);
        if (e + 16 < c) v.z = __ldg(row + e + 16);
        if (e + 24 < c) v.w = __ldg(row + e + 24);
    } else {
        const int e = k + 4 * sub;
        if (e < c) v = __ldg(reinterpret_cast<const int4 *>(row + e));
        if (e + 1 >= c) v.y = -1;
        if (e + 2 >= c) v.z = -1;
        if (e + 3 >= c) v.w = -1;
    }
    return v;
}

// TPP lanes share one particle; a block takes a.particles particles of one
// system in rounds of kLJBlock / TPP.
//
// What bounds it: instruction issue and the latency of the gathers of neighbour
// positions (N = 262,144, two lanes: 64% of the issue rate, L1 data pipe 72%,
// long-scoreboard stalls first).  So a pair takes no branch but the one for
// pairs across a face: every pair's terms are formed and added by predicate.  The next
// particle is looked up one round ahead and a row's next chunk one chunk ahead.
//
// The energy of a particle is the sum of two FP32 sums, of entries 8 k .. 8 k + 3
// and of 8 k + 4 .. 8 k + 7 in order (two lanes per particle, the default), and U
// adds those FP32 sums in FP64.  SPREAD gives the particle 8 lanes and keeps
// those sums: lanes 0 to 3 (4 to 7) all add the first (second) one's terms, in
// order, from each other's registers.
//
// FP64 runs at about two operations per cycle and SM: an instruction of a warp
// takes 16 cycles.  Every lane's FP32 sums of gradient terms enter FP64 by
// themselves: even lanes add up the particle's dU/deps terms and odd ones its
// dU/dsig terms, in the same instructions.  GRAD = false leaves them out where
// the caller asked for neither.
template <int T, int TPP, bool GRAD, bool SPREAD>
__global__ void __launch_bounds__(kLJBlock, T <= 2 ? QBVH_LJ_MIN_BLOCKS : 1)
lj_forward_kernel(const __grid_constant__ LJArgs a)
{
    static_assert(!SPREAD || TPP == 8, "SPREAD: 8 lanes per particle");
    constexpr int NP = 1 + 2 * T * T;
    constexpr int TG = GRAD ? T : 1;
    constexpr int SETS = TPP == 1 ? 2 : 1;   // one lane keeps both gradients' sums
    // lanes of a particle that keep FP64 sums: its other lanes add to theirs in every
    // round, or (16 and 32 lanes, where that is four and five more additions a round) all
    // lanes keep their own to the end.  Two types, N = 300,000, 4 / 8 / 16 / 32 lanes:
    // 149 / 184 / 252 / 422 us the first way, 153 / 182 / 231 / 317 the second.
    constexpr int KEEP = TPP <= 8 ? (TPP == 1 ? 1 : 2) : TPP;
    __shared__ LJParams s_par[T * T];
    __shared__ double s_red[kLJBlock / 32][NP];
    const int tid = threadIdx.x;
    if (tid < T * T) s_par[tid] = lj_params(a.eps[tid], a.sig[tid], a.rc2[tid]);
    __syncthreads();
    const int sys = a.blk_sys[blockIdx.x];
    const SysInfo sy = a.sys[sys];
    const int sub = tid % TPP;
    const int begin = a.blk_first[blockIdx.x];
    const int end = min(begin + a.particles, sy.offset + sy.count);
    double v = 0.0, acc[SETS][TG * TG];
#pragma unroll
    for (int h = 0; h < SETS; ++h)
#pragma unroll
        for (int q = 0; q < TG * TG; ++q) acc[h][q] = 0.0;
    // position in the walk order: Z-order when the tree's order is given, so
    // that a block's particles are close and their neighbours' positions are
    // shared in L1; systems occupy the same index range in both orders
    int sidx = begin + tid / TPP;
    int i = sidx < end ? (a.order ? __ldg(a.order + sidx) : sidx) : -1;
    for (int base = begin; base < end; base += kLJBlock / TPP) {
        sidx += kLJBlock / TPP;
        const int inext = sidx < end ? (a.order ? __ldg(a.order + sidx) : sidx) : -1;
        float e = 0.f, fx = 0.f, fy = 0.f, fz = 0.f;
        float gE[TG], gS[TG];
#pragma unroll
        for (int b = 0; b < TG; ++b) gE[b] = gS[b] = 0.f;
        int ta = 0;
        if (i >= 0) {
            const int c = min(__ldg(a.counts + i), a.cap);
            const int *row = a.rows + (size_t)i * a.cap;
            const float4 pi = __ldg(a.pos + i);
            ta = T > 1 ? __float_as_int(pi.w) : 0;
            ta = ta < 0 ? 0 : (ta >= T ? T - 1 : ta);
            int4 next = row_chunk<SPREAD>(row, 0, sub, c);
            for (int k = 0; k < c; k += 4 * TPP) {
                const int jj[4] = {next.x, next.y, next.z, next.w};
                if (k + 4 * TPP < c) next = row_chunk<SPREAD>(row, k + 4 * TPP, sub, c);
                float4 pp[4];
                bool ok[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    ok[u] = (unsigned)jj[u] < (unsigned)a.n;
                    pp[u] = __ldg(a.pos + (ok[u] ? jj[u] : i));
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (SPREAD && k + 8 * u >= c) break;   // the same for the particle's lanes
                    const float4 pj = pp[u];
                    int tb = T > 1 ? __float_as_int(pj.w) : 0;
                    tb = tb < 0 ? 0 : (tb >= T ? T - 1 : tb);
                    const LJPairGeom gm = lj_pair_geom(pi, pj, sy.L, sy.Linv);
                    const LJParams &par = s_par[ta * T + tb];
                    const bool in = ok[u] && gm.r2 < par.rc2;
                    const LJPairTerms t = lj_pair_terms<QBVH_LJ_FAST_RCP>(gm.vr2, par);
                    if (SPREAD) {
                        const unsigned group = 0xFFu << (tid & 24);
                        const float term = in ? t.uE : 0.f;
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const int src = (tid & 28) | r;
                            const float x = __shfl_sync(group, term, src);
                            const float eps = T > 1 ? __shfl_sync(group, par.eps, src) : par.eps;
                            if (x != 0.f) e = fmaf(eps, x, e);
                        }
                    } else {
                        e = in ? fmaf(par.eps, t.uE, e) : e;
                    }
                    fx = in ? fmaf(-t.w, gm.vx, fx) : fx;
                    fy = in ? fmaf(-t.w, gm.vy, fy) : fy;
                    fz = in ? fmaf(-t.w, gm.vz, fz) : fz;
                    if (GRAD) {
#pragma unroll
                        for (int b = 0; b < TG; ++b) {
                            gE[b] = b == tb && in ? gE[b] + t.uE : gE[b];
                            gS[b] = b == tb && in ? gS[b] + t.gs : gS[b];
                        }
                    }
                }
            }
        }
        // per-particle results: FP32 sums over the group's lanes
        float ei = e;
        if (SPREAD) {
            ei += __shfl_xor_sync(0xFFFFFFFFu, ei, 4);
        } else {
#pragma unroll
            for (int o = TPP / 2; o > 0; o >>= 1) ei += __shfl_xor_sync(0xFFFFFFFFu, ei, o);
        }
#pragma unroll
        for (int o = TPP / 2; o > 0; o >>= 1) {
            fx += __shfl_xor_sync(0xFFFFFFFFu, fx, o);
            fy += __shfl_xor_sync(0xFFFFFFFFu, fy, o);
            fz += __shfl_xor_sync(0xFFFFFFFFu, fz, o);
        }
        if (i >= 0 && sub == 0) {
            if (a.e) a.e[i] = 0.5f * ei;
            if (a.F) {
                a.F[3 * (size_t)i] = fx;
                a.F[3 * (size_t)i + 1] = fy;
                a.F[3 * (size_t)i + 2] = fz;
            }
        }
        // FP64 sums of the energy (a lane's FP32 sum; SPREAD: lanes 0 and 4 hold the
        // two) and of the lanes' parameter-gradient terms; the factor 1/2 comes at the end
        if (!SPREAD || (sub & 3) == 0) v += (double)e;
        if (GRAD) {
#pragma unroll
            for (int h = 0; h < SETS; ++h) {
#pragma unroll
                for (int b = 0; b < TG; ++b) {
                    double g = (double)((TPP == 1 ? h == 1 : (sub & 1) != 0) ? gS[b] : gE[b]);
                    if (TPP > 1) g += (double)__shfl_xor_sync(0xFFFFFFFFu, (sub & 1) ? gE[b] : gS[b], 1);
#pragma unroll
                    for (int o = TPP / 2; TPP > 1 && o >= KEEP; o >>= 1) g += __shfl_xor_sync(0xFFFFFFFFu, g, o);
#pragma unroll
                    for (int t = 0; t < TG; ++t)
                        if (t == ta && sub < KEEP) acc[h][t * TG + b] += g;
                }
            }
        }
        i = inext;
    }
    const int lane = tid & 31, warp = tid >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    if (lane == 0) s_red[warp][0] = v;
    if (GRAD) {
#pragma unroll
        for (int h = 0; h < SETS; ++h) {
#pragma unroll
            for (int q = 0; q < TG * TG; ++q) {
                double x = acc[h][q];
#pragma unroll
                for (int o = 16; o >= (KEEP < TPP || TPP == 1 ? TPP : 2); o >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, o);
                // lane 0: dU/deps; lane 1 (one lane per particle: the second set): dU/dsig
                if (TPP == 1 ? lane == 0 : lane < 2) s_red[warp][(1 + (TPP == 1 ? h : lane) * T * T + q) % NP] = x;
            }
        }
    }
    __syncthreads();
    for (int q = tid; q < (GRAD ? NP : 1); q += kLJBlock) {
        double x = 0.0;
        for (int w = 0; w < kLJBlock / 32; ++w) x += s_red[w][q];
        a.partials[(size_t)blockIdx.x * NP + q] = 0.5 * x;
    }
}

// One block per system and value: fixed-order FP64 sum of the block records.
// Thread t sums records t, t + kFinThreads, ... in order, then the warps and the
// block add up in a fixed order: the same order on every call.  (All values of a
// system in one block, ten barriers each, took 14 to 40 us.)
constexpr int kFinThreads = 256;
// Without a block table (sys_blk_start == nullptr) one system owns records
// [0, n_blocks).
__global__ void __launch_bounds__(kFinThreads) lj_finalize_kernel(const double *partials, const int *sys_blk_start,
                                                                  int np, int T, double *U, double *dE, double *dS,
                                                                  int n_blocks = 0)
{
    __shared__ double s[kFinThreads / 32];
    const int sys = blockIdx.x, q = blockIdx.y;
    const int t = threadIdx.x;
    const int b0 = sys_blk_start ? sys_blk_start[sys] : 0;
    const int b1 = sys_blk_start ? sys_blk_start[sys + 1] : n_blocks;
    double x = 0.0;
#pragma unroll 8
    for (int b = b0 + t; b < b1; b += kFinThreads) x += partials[(size_t)b * np + q];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, o);
    if ((t & 31) == 0) s[t >> 5] = x;
    __syncthreads();
    if (t != 0) return;
    double tot = 0.0;
    for (int w = 0; w < kFinThreads / 32; ++w) tot += s[w];
    if (q == 0) U[sys] = tot;
    else if (q <= T * T) { if (dE) dE[(size_t)sys * T * T + (q - 1)] = tot; }
    else if (dS) dS[(size_t)sys * T * T + (q - 1 - T * T)] = tot;
}

__global__ void lj_backward_pos_kernel(const double *g, const float *F, float *gpos, int n, int n_sys,
                                       const int *sys_off)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = n_sys - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(sys_off + mid) <= i) lo = mid; else hi = mid - 1;
    }
    const float gs = (float)g[lo];
    for (int d = 0; d < 3; ++d) gpos[3 * (size_t)i + d] = -gs * F[3 * (size_t)i + d];
}

__global__ void lj_backward_param_kernel(const double *g, const double *dE, const double *dS, float *geps,
                                         float *gsig, int n_sys, int TT)
{
    const int q = threadIdx.x;
    if (q >= TT) return;
    double xe = 0.0, xs = 0.0;
    for (int k = 0; k < n_sys; ++k) {
        if (dE) xe += g[k] * dE[(size_t)k * TT + q];
        if (dS) xs += g[k] * dS[(size_t)k * TT + q];
    }
    if (geps) geps[q] = (float)xe;
    if (gsig) gsig[q] = (float)xs;
}

__global__ void pack_kernel(const float *xyz, const int *types, int n, float4 *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int t = types ? types[i] : 0;
    out[i] = make_float4(xyz[3 * (size_t)i], xyz[3 * (size_t)i + 1], xyz[3 * (size_t)i + 2], __int_as_float(t));
}

}  // namespace

// Particles per block: 256, halved down to one round while the grid would hold
// fewer than 36 blocks per SM.  (Seven stay resident.  18 / 36 / 72 blocks per SM,
// microseconds: one type, N = 131,072 53 / 52 / 55, 1,000,000 220 / 212 / 221; two types
// with gradients, 1,000,000 302 / 300 / 321, 2,097,152 577 / 577 / 588.)
int lj_particles_per_block(int n, int tpp)
{
    const int round = kLJBlock / (tpp == 0 ? 8 : tpp);
    int p = 256;
    while (p > round && n / p < 152 * 36) p >>= 1;
    return p;
}

// 8 lanes per particle that keep the sums of two, where two (the default) would
// leave most of the GPU idle: two-type gradients of 2 x 2827 particles 29 -> 19 us,
// N = 30,011 33 us either way, N = 131,072 with r = 1.12 27 -> 50 us.
bool lj_spread(int n) { return n < 30000; }

template <int T, int TPP, bool SPREAD>
static void launch_lj_tpp(const LJArgs &a, cudaStream_t s)
{
    if (a.dE || a.dS) lj_forward_kernel<T, TPP, true, SPREAD><<<a.n_blocks, kLJBlock, 0, s>>>(a);
    else lj_forward_kernel<T, TPP, false, SPREAD><<<a.n_blocks, kLJBlock, 0, s>>>(a);
}

template <int T>
static void launch_lj_t(const LJArgs &a, cudaStream_t s)
{
    switch (a.tpp) {
    case 0: launch_lj_tpp<T, 8, true>(a, s); break;
    case 1: launch_lj_tpp<T, 1, false>(a, s); break;
    case 2: launch_lj_tpp<T, 2, false>(a, s); break;
    case 4: launch_lj_tpp<T, 4, false>(a, s); break;
    case 8: launch_lj_tpp<T, 8, false>(a, s); break;
    case 16: launch_lj_tpp<T, 16, false>(a, s); break;
    default: launch_lj_tpp<T, 32, false>(a, s); break;
    }
}

void launch_lj_forward(const LJArgs &a, cudaStream_t s)
{
    if (a.n_blocks > 0) {
        switch (a.n_types) {
        case 1: launch_lj_t<1>(a, s); break;
        case 2: launch_lj_t<2>(a, s); break;
        case 3: launch_lj_t<3>(a, s); break;
        case 4: launch_lj_t<4>(a, s); break;
        case 5: launch_lj_t<5>(a, s); break;
        case 6: launch_lj_t<6>(a, s); break;
        case 7: launch_lj_t<7>(a, s); break;
        default: launch_lj_t<8>(a, s); break;
        }
    }
    const int T = a.n_types, np = 1 + 2 * T * T;
    const dim3 grid(a.n_sys, a.dE || a.dS ? np : 1);
    lj_finalize_kernel<<<grid, kFinThreads, 0, s>>>(a.partials, a.sys_blk_start, np, T, a.U, a.dE, a.dS);
}

void launch_lj_finalize_one(const double *partials, int n_blocks, double *U, double *dE, double *dS,
                            cudaStream_t s)
{
    lj_finalize_kernel<<<dim3(1, dE || dS ? 3 : 1), kFinThreads, 0, s>>>(partials, nullptr, 3, 1, U, dE, dS, n_blocks);
}

void launch_lj_backward(const double *g, const float *F, const double *dE, const double *dS, float *gpos,
                        float *geps, float *gsig, int n, int n_sys, int n_types, const SysInfo *sys,
                        const int *sys_off, cudaStream_t s)
{
    (void)sys;
    if (gpos && F && n > 0) lj_backward_pos_kernel<<<(n + 255) / 256, 256, 0, s>>>(g, F, gpos, n, n_sys, sys_off);
    if (geps || gsig) lj_backward_param_kernel<<<1, 64, 0, s>>>(g, dE, dS, geps, gsig, n_sys, n_types * n_types);
}

void launch_pack(const float *xyz, const int *types, int n, float4 *out, cudaStream_t s)
{
    if (n > 0) pack_kernel<<<(n + 255) / 256, 256, 0, s>>>(xyz, types, n, out);
}

}  // namespace qbvh
