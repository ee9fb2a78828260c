// batch.cu -- multi-scene frame step of the VIPER library (sm_103a).
//
// viper_batch_step advances many scenes by one frame with one launch sequence
// for all of them.  Each kernel's grid is the concatenation of the scenes'
// grids for that kernel kind; a CTA finds its scene with one barrier count
// over the kind's block offsets and stages the scene's parameters (the same
// Params the one-scene kernels take by value) in shared memory.  The
// per-element work is the one-scene kernels' device code (phases.cuh), so a
// scene computes the same thing alone and in a batch.
//
// Per substep, contact path (pills and/or half-planes), I >= 1 iterations:
//   velocity update of the previous substep + prediction |
//   [grid (a cluster of CTAs per scene: cull, bounds, cut, counts, scan, scatter) |
//   pair search] beside [sweep 0, on a second stream] |
//   contact | {sweep | contact} x (I - 1)
// and one velocity update after the last substep: S (2 I + 3) + 1 launches (three
// more a substep where a scene is too large for the cluster's grid; without pills no
// grid and search, and the update, the prediction and sweep 0 in one launch; bundles
// add one).  Without contacts: one launch for all substeps.  After the
// substeps one launch builds the skinning frames, hands the bone pose on and
// mirrors the error word to the host; one more skins every mesh.
//
// The per-call table (scene parameters, block offsets, bone poses) is written
// into pinned staging and uploaded with one copy; two staging buffers let the
// host fill the next call's table while the previous call runs.
#include <string.h>

#include <algorithm>
#include <map>
#include <vector>

#include "phases.cuh"

namespace viper {

enum BatchKind : int { K_ELEM = 0, K_PILL, K_EMIT, K_SCAN, K_GRID, K_ROD, K_CONTACT, K_END, K_MESH, K_BUNDLE, K_WARM, K_KINDS };

// One scene of a batched frame, as the device sees it.
struct BatchScene {
    Params P;  // h, inv_h, inv_h2 of this frame; bq1 / bt1 point at the frame's target pose
    const float4 *LQ, *LC;
    const int *sperm;
    float4 *frames;
    const float4 *rest;
    const int4 *idx;
    const float4 *w;
    float4 *out;
    float4 *bq0, *bq1_own;  // the scene's previous / target pose buffers
    float *bt0, *bt1_own;
    int *herr;              // device address of the scene's mapped error mirror
    int n_mesh, n_bones, pills, pad;
};

struct BatchArgs {
    const BatchScene *sc;
    const int *off;  // K_KINDS rows of n + 1 block offsets
    int n;
};

constexpr int kElemThreads = 256, kEmitWarpsB = 8, kScanThreadsB = 1024, kScanPerB = 16;

// Scene of this CTA for `kind` (the last scene whose first block is <= blockIdx.x),
// staged in shared memory; local = block index within the scene, nblk = its block count.
// Kernels are launched with programmatic dependent launch (see pdl_wait): this
// prologue overlaps the predecessor kernel.
__device__ __forceinline__ void batch_scene(const BatchArgs &A, int kind, BatchScene &sb, int &local, int &nblk)
{
    __shared__ int s_lo, s_hi;
    const int *o = A.off + kind * (A.n + 1);
    const int b = blockIdx.x;
    int cnt = 0;
    for (int base = 0; base < A.n; base += blockDim.x) {
        const int t = base + threadIdx.x;
        cnt += __syncthreads_count(t < A.n && o[t] <= b);
    }
    const int s = cnt - 1;  // o[0] = 0 <= b, so 0 <= s < n
    if (threadIdx.x == 0) {
        s_lo = o[s];
        s_hi = o[s + 1];
    }
    const int *src = reinterpret_cast<const int *>(A.sc + s);
    int *dst = reinterpret_cast<int *>(&sb);
    for (int k = threadIdx.x; k < (int)(sizeof(BatchScene) / 4); k += blockDim.x) dst[k] = src[k];
    __syncthreads();
    local = b - s_lo;
    nblk = s_hi - s_lo;
}

__device__ __forceinline__ void batch_enter(const BatchArgs &A, int kind, BatchScene &sb, int &local, int &nblk)
{
    batch_scene(A, kind, sb, local, nblk);
    // Everything above reads only the call's table, uploaded before the first
    // kernel of the call; the scene state is read after the predecessor kernel
    // has finished.  The successor is released once every CTA got here.
    pdl_wait();
    pdl_trigger();
}

// ---------------------------------------------------------------- substep kernels
// Prediction (Sec. 6) of every vertex and segment; clears the scene's
// broadphase bounds for this substep's merge.
__global__ void __launch_bounds__(kElemThreads) batch_predict_kernel(BatchArgs A, float tau)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_ELEM, sb, local, nblk);
    const Params &P = sb.P;
    if (sb.pills && local == 0 && threadIdx.x < 8) P.bounds[threadIdx.x] = 0u;
    const int i = local * blockDim.x + threadIdx.x;
    if (i < P.nv)
        predict_vertex_at(P, i, tau, sb.pills != 0, false);
    else if (i < P.nv + P.ns)
        predict_segment_at(P, i - P.nv, false);
}

__global__ void __launch_bounds__(kElemThreads) batch_bounds_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_PILL, sb, local, nblk);
    const Params &P = sb.P;
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY}, mr = 0.f;
    const int g = local * blockDim.x + threadIdx.x;
    if (g < P.ns) bound_pill(P, g, mn, mx, mr);
    merge_bounds(P, mn, mx, mr);
}

__global__ void __launch_bounds__(kElemThreads) batch_count_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_PILL, sb, local, nblk);
    const Params &P = sb.P;
    bool ok;
    const Grid G = make_grid(P, ok);
    if (local == 0 && threadIdx.x == 0) {
        *P.grid = G;
        *P.npairs = 0;
        if (!ok) atomicOr(P.err, ERR_NONFINITE);
    }
    const int g = local * blockDim.x + threadIdx.x;
    if (g < P.ns) count_pill(P, G, g);
}

// Exclusive scan of the scene's cell counts over the cells its grid spans, by
// one CTA, 16 cells per thread per round; cell_start[cells] = number of pills.
__global__ void __launch_bounds__(kScanThreadsB) batch_scan_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    __shared__ int ws[33];
    int local, nblk;
    batch_enter(A, K_SCAN, sb, local, nblk);
    const int n = grid_cells(sb.P.grid, sb.P.table);
    const int *cc = sb.P.cell_count;
    int *cs = sb.P.cell_start;
    int carry = 0;
    for (int base = 0; base < n; base += kScanThreadsB * kScanPerB) {
        const int b0 = base + threadIdx.x * kScanPerB;
        int v[kScanPerB], s = 0;
#pragma unroll
        for (int k = 0; k < kScanPerB; ++k) {
            v[k] = (b0 + k < n) ? cc[b0 + k] : 0;
            s += v[k];
        }
        int tot;
        int off = block_excl_scan(s, ws, &tot) + carry;
#pragma unroll
        for (int k = 0; k < kScanPerB; ++k) {
            if (b0 + k < n) cs[b0 + k] = off;
            off += v[k];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) cs[n] = carry;
}

__global__ void __launch_bounds__(kElemThreads) batch_scatter_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_PILL, sb, local, nblk);
    const Params &P = sb.P;
    const int g = local * blockDim.x + threadIdx.x;
    if (g < P.ns) {
        const int cell = P.cell_of[g];
        scatter_pill(P, g, cell, P.cell_start[cell]);
    }
}

// Candidate pairs: a warp per oversized pill (with the cluster's grid), then L
// lanes per pill (see emit_big, emit_pills).
template <int L>
__global__ void __launch_bounds__(32 * kEmitWarpsB) batch_emit_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    __shared__ int buf[kEmitWarpsB][kEmitBuf];
    int local, nblk;
    batch_enter(A, K_EMIT, sb, local, nblk);
    const Params &P = sb.P;
    const Grid G = *P.grid;
    if (G.pad) return;  // no valid grid: no candidates (uniform over the CTA)
    const int wib = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31, warp = local * kEmitWarpsB + wib, nwarps = nblk * kEmitWarpsB;
    const int n = P.cell_start[grid_cells(&G, P.table)];  // pills in the cells
    const unsigned int big = big_threshold(G.b_cut);
    const int nb = G.b_cut < kRadBins - 1 ? min(P.bp_hist[kRadBins], P.big_cap) : 0;
    for (int i = warp; i < nb; i += nwarps) emit_big(P, G, big, i, buf[wib], lane);
    emit_pills<L>(P, G, big, n, warp, nwarps, buf[wib], lane);
}

// ---------------------------------------------------------------- one scene's grid by one cluster
__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_ctas()
{
    unsigned r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Every thread of the cluster calls both; they order shared and global memory between its CTAs.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}
// Address of shared variable p in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned in_cta(const void *p, unsigned rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;"
        : "=r"(r)
        : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_store(unsigned addr, unsigned v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ int cluster_load(unsigned addr)
{
    int v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ int cluster_add(unsigned addr, int v)
{
    int r;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(r) : "r"(addr), "r"(v) : "memory");
    return r;
}

// One scene's broadphase grid by one cluster of CTAs: bounding spheres and their
// bounds, the grid, cell counts, the exclusive cell scan into cell_start, and
// the scatter into cell order with the sphere / group copies.
//
// Pills that can touch no pill of another group are left out first (scenes of up
// to kGridGroupsMax groups): a group's box, enlarged well above the rounding of
// spheres_overlap, bounds its pills' spheres; where two groups' boxes meet, a
// pill of either can only touch the other's inside the meeting of the boxes; and
// a pill stays if it reaches the box around its group's meetings.  A rig's
// muscles lie side by side: of 6,910 pills 24 stay, where the cells (as wide as
// the largest pill, nine times the smallest) held 180 candidates a pill, nearly
// all of the pill's own muscle.
//
// Where at most kGridFew stay, they are put in one cell, and the pair search tests
// them all; the steps below are left out.
//
// The build is a chain of dependent phases, too short for a launch each and too
// long for one CTA (10,080 pills: 38.5 us by one CTA of 512 threads, 12 by eight).
// The cluster splits the pills into slices and the cells into ranges of 2^sh,
// one of each per CTA, all in shared memory: spheres and the pills' cells in
// their slice, counts and starts in the range's owner.  Counting a pill returns
// its place within its cell, so that the scatter needs no second pass of atomics.
// The CTAs meet five times (boxes, bounds, counts, range totals, end).
// Dynamic shared memory: slice_cap spheres, cells (first the pills' vertices) and
// places (first their groups), cells_cap cell counts (the table's share of a CTA, a
// power of two), and per group this CTA's and the scene's box.
constexpr int kGridThreads = 512, kGridClusterMax = 8, kGridCellsMax = 16384, kGridSliceMax = 5120;
constexpr int kGridMaxPills = kGridClusterMax * kGridSliceMax;  // 40,960: table of 131,072 cells = 8 x kGridCellsMax
constexpr int kGridGroupsMax = 512, kGridFew = 128;
inline int grid_smem_bytes(int cells_cap, int slice_cap, int groups_cap)
{
    return (16 + 4 + 4) * slice_cap + 4 * cells_cap + 64 * groups_cap;
}
static_assert((16 + 4 + 4) * kGridSliceMax + 4 * kGridCellsMax + 64 * kGridGroupsMax + 6144 <= 227 * 1024,
              "the largest scene's grid fits a CTA's shared memory (6 KB of it static)");

// Half-width of the box of sphere sp in the cull: its radius and a margin far above
// the rounding of the box and of spheres_overlap.
__device__ __forceinline__ float cull_reach(float4 sp)
{
    return 1.0078125f * fabsf(sp.w) + 1e-6f * (fabsf(sp.x) + fabsf(sp.y) + fabsf(sp.z));
}

// Whether all bounds are finite, as make_grid_from requires them.
__device__ __forceinline__ bool finite_bounds(const unsigned *bounds)
{
    bool ok = isfinite(2.f * ord_dec(bounds[6]) * 1.00390625f);
    for (int c = 0; c < 3; ++c) {
        const float lo = -ord_dec(bounds[c]), hi = ord_dec(bounds[3 + c]);
        ok = ok && isfinite(lo) && isfinite(hi) && hi >= lo;
    }
    return ok;
}

// Without a result: an addition whose result is dropped waits for the one before it.
__device__ __forceinline__ void cluster_max(unsigned addr, unsigned v)
{
    asm volatile("red.shared::cluster.max.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_count(unsigned addr, int v)
{
    asm volatile("red.shared::cluster.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// A group's box in the table: the corners as unsigned numbers that order as the
// floats do (ord_enc), the low one inverted so that both grow with the box; zero is
// the empty box, which meets none.
struct __align__(16) GroupBox {
    unsigned lo[4], hi[4];  // the fourth entries only align
};

// Sphere sp of a pill of group grp into the box table; the lanes `act` call it
// together, one addition per group.
__device__ __forceinline__ void box_add(GroupBox *box, unsigned act, int grp, float4 sp)
{
    const unsigned peers = __match_any_sync(act, grp);
    const float r = cull_reach(sp);
    const bool in = isfinite(sp.x + sp.y + sp.z + r);  // no pair has a sphere that is not
    const float c[3] = {sp.x, sp.y, sp.z};
    unsigned lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k] = __reduce_max_sync(peers, in ? ~ord_enc(c[k] - r) : 0u);
        hi[k] = __reduce_max_sync(peers, in ? ord_enc(c[k] + r) : 0u);
    }
    if ((threadIdx.x & 31) == __ffs(peers) - 1)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            atomicMax(&box[grp].lo[k], lo[k]);
            atomicMax(&box[grp].hi[k], hi[k]);
        }
}

// The box around group a's meetings with the other groups' boxes, by one warp,
// written to hot as floats (empty: low above high).
__device__ __forceinline__ void hot_box(const GroupBox *box, int groups, int a, GroupBox *hot, int lane)
{
    const uint4 *tab = reinterpret_cast<const uint4 *>(box);
    const uint4 al = tab[2 * a], ah = tab[2 * a + 1];
    float hl[3] = {INFINITY, INFINITY, INFINITY}, hh[3] = {-INFINITY, -INFINITY, -INFINITY};
    bool any = false;
    for (int b = lane; b < groups; b += 32) {
        const uint4 bl = tab[2 * b], bh = tab[2 * b + 1];
        if (b == a || ~al.x > bh.x || ~al.y > bh.y || ~al.z > bh.z || ~bl.x > ah.x || ~bl.y > ah.y || ~bl.z > ah.z)
            continue;
        any = true;
        const unsigned l[3] = {~min(al.x, bl.x), ~min(al.y, bl.y), ~min(al.z, bl.z)};
        const unsigned h[3] = {min(ah.x, bh.x), min(ah.y, bh.y), min(ah.z, bh.z)};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            hl[k] = fminf(hl[k], ord_dec(l[k]));
            hh[k] = fmaxf(hh[k], ord_dec(h[k]));
        }
    }
    if (__any_sync(0xffffffffu, any))
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                hl[k] = fminf(hl[k], __shfl_xor_sync(0xffffffffu, hl[k], o));
                hh[k] = fmaxf(hh[k], __shfl_xor_sync(0xffffffffu, hh[k], o));
            }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            hot->lo[k] = __float_as_uint(hl[k]);
            hot->hi[k] = __float_as_uint(hh[k]);
        }
}

__global__ void __launch_bounds__(kGridThreads, 2)
    batch_grid_kernel(BatchArgs A, int cells_cap, int slice_cap, int groups_cap)
{
    __shared__ BatchScene sb;
    __shared__ unsigned int s_bounds[8], s_kept[8];     // of all pills, of those that stay
    __shared__ unsigned int s_all[kGridClusterMax][8];  // the CTAs' bounds
    __shared__ unsigned int s_all_kept[kGridClusterMax][8];
    __shared__ int s_tot[kGridClusterMax];              // the ranges' totals
    __shared__ int s_stay;                              // this CTA's pills that stay
    __shared__ int s_hist[kRadBins + 33], s_hist_all[kRadBins];  // radii, for the cut (see choose_cut)
    __shared__ int ws[33];
    extern __shared__ __align__(16) unsigned char s_dyn[];
    float4 *s_sph = reinterpret_cast<float4 *>(s_dyn);
    int *s_cell = reinterpret_cast<int *>(s_sph + slice_cap);
    int *s_place = s_cell + slice_cap;
    int *s_count = s_place + slice_cap;
    GroupBox *s_own = reinterpret_cast<GroupBox *>(s_count + cells_cap), *s_box = s_own + groups_cap;
    unsigned *own_words = reinterpret_cast<unsigned *>(s_own), *box_words = reinterpret_cast<unsigned *>(s_box);
    int local, nblk;
    batch_scene(A, K_GRID, sb, local, nblk);
    const Params &P = sb.P;
    const int t = threadIdx.x, bd = blockDim.x, ns = P.ns;
    const unsigned rank = cluster_rank(), ctas = cluster_ctas();
    const int per = (ns + (int)ctas - 1) / (int)ctas;
    const int g0 = min((int)rank * per, ns), n = min(per, ns - g0);  // this CTA's pills [g0, g0 + n)
    // before the predecessor has finished: what does not depend on the state
    const int groups = P.n_groups <= groups_cap ? P.n_groups : 0;  // 0: every pill stays
    if (t < 8) s_bounds[t] = s_kept[t] = 0u;
    if (t == 0) s_stay = 0;
    for (int c = t; c < cells_cap; c += bd) s_count[c] = 0;
    for (int c = t; c < kRadBins; c += bd) s_hist[c] = s_hist_all[c] = 0;
    for (int c = t; c < 8 * groups; c += bd) own_words[c] = box_words[c] = 0u;
    for (int i = t; i < n; i += bd) {
        s_cell[i] = P.seg_v0[g0 + i];
        s_place[i] = P.seg_group[g0 + i];
    }
    __syncthreads();
    cluster_arrive();
    pdl_wait();
    pdl_trigger();

    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY}, mr = 0.f;
    {
        const float4 *xp = P.Xpred;
        const float *rbar = P.bp_rbar;
        const size_t rs = (size_t)P.bp_rbar_stride;
        for (int base = 0; base < n; base += 4 * bd) {  // 4 pills per thread and batch, loads issued together
            float4 xa[4], xb[4];
            float ra[4], rb[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = base + k * bd + t;
                const size_t a = i < n ? s_cell[i] : 0;
                xa[k] = xp[a];
                xb[k] = xp[a + 1];
                ra[k] = rbar[a * rs];
                rb[k] = rbar[(a + 1) * rs];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = base + k * bd + t;
                const unsigned act = __ballot_sync(0xffffffffu, i < n);
                if (i >= n) continue;
                const float4 sp = pill_sphere(xa[k], ra[k], xb[k], rb[k]);
                s_sph[i] = sp;
                if (groups)
                    box_add(s_own, act, s_place[i], sp);
                else
                    hist_add(s_hist, act, sp.w);
                mn[0] = fminf(mn[0], sp.x); mn[1] = fminf(mn[1], sp.y); mn[2] = fminf(mn[2], sp.z);
                mx[0] = fmaxf(mx[0], sp.x); mx[1] = fmaxf(mx[1], sp.y); mx[2] = fmaxf(mx[2], sp.z);
                mr = fmaxf(mr, fabsf(sp.w));
            }
        }
    }
    merge_bounds_to(s_bounds, mn, mx, mr);
    __syncthreads();
    cluster_wait();  // every CTA of the cluster has started
    for (int k = t; k < 8 * (int)ctas; k += bd) cluster_store(in_cta(&s_all[rank][k & 7], k >> 3), s_bounds[k & 7]);
    for (int k = t; k < 8 * groups; k += bd)
        if (own_words[k])
            for (unsigned r = 0; r < ctas; ++r) cluster_max(in_cta(box_words + k, r), own_words[k]);
    auto share_hist = [&]() {
        for (int k = t; k < kRadBins; k += bd)
            if (s_hist[k])
                for (unsigned r = 0; r < ctas; ++r) cluster_count(in_cta(s_hist_all + k, r), s_hist[k]);
    };
    if (!groups) share_hist();
    if (rank == 0 && t == 0) P.bp_hist[kRadBins] = 0;  // oversized pills listed
    cluster_sync();  // bounds and boxes, or bounds and histogram, exchanged
    if (t < 8) {
        unsigned int m = 0u;
        for (unsigned r = 0; r < ctas; ++r) m = max(m, s_all[r][t]);
        s_bounds[t] = m;
    }
    __syncthreads();
    bool ok;
    Grid G;
    if (groups) {
        // the groups of this CTA's pills: their meetings with the others, then the pills that reach them
        const int lane = t & 31;
        for (int a = t >> 5; a < groups; a += bd >> 5)
            if (s_own[a].hi[0]) hot_box(s_box, groups, a, s_own + a, lane);
        __syncthreads();
        float kn[3] = {INFINITY, INFINITY, INFINITY}, kx[3] = {-INFINITY, -INFINITY, -INFINITY}, kr = 0.f;
        for (int base = 0; base < n; base += bd) {
            const int i = base + t;
            bool stays = false;
            float4 sp;
            if (i < n) {
                sp = s_sph[i];
                const float r = cull_reach(sp);
                const GroupBox &hot = s_own[s_place[i]];
                const float4 l = *reinterpret_cast<const float4 *>(hot.lo), h = *reinterpret_cast<const float4 *>(hot.hi);
                stays = sp.x - r <= h.x && sp.y - r <= h.y && sp.z - r <= h.z && sp.x + r >= l.x && sp.y + r >= l.y &&
                        sp.z + r >= l.z;
                s_cell[i] = stays ? 0 : -1;
            }
            const unsigned m = __ballot_sync(0xffffffffu, stays);
            int first = 0;
            if (lane == 0 && m) first = atomicAdd(&s_stay, __popc(m));
            first = __shfl_sync(0xffffffffu, first, 0);
            if (!stays) continue;
            s_place[i] = first + __popc(m & ((1u << lane) - 1u));  // among this CTA's
            kn[0] = fminf(kn[0], sp.x); kn[1] = fminf(kn[1], sp.y); kn[2] = fminf(kn[2], sp.z);
            kx[0] = fmaxf(kx[0], sp.x); kx[1] = fmaxf(kx[1], sp.y); kx[2] = fmaxf(kx[2], sp.z);
            kr = fmaxf(kr, fabsf(sp.w));
        }
        __syncwarp();
        merge_bounds_to(s_kept, kn, kx, kr);
        __syncthreads();
        if (t < 8 * (int)ctas)
            cluster_store(in_cta(&s_all_kept[rank][t & 7], t >> 3), (t & 7) == 7 ? (unsigned)s_stay : s_kept[t & 7]);
        cluster_sync();
        ok = finite_bounds(s_bounds);  // of all pills, as without the cull
        int total = 0, before = 0;
        for (unsigned r = 0; r < ctas; ++r) {
            if (r == rank) before = total;
            total += (int)s_all_kept[r][7];
        }
        if (total <= kGridFew) {  // few stay: one cell of all, every pair tested
            for (int i = t; i < n; i += bd)
                if (s_cell[i] >= 0) {
                    const int pos = before + s_place[i];
                    P.cell_pills[pos] = g0 + i;
                    P.cell_sph[pos] = s_sph[i];
                    P.cell_grp[pos] = P.seg_group[g0 + i];
                }
            if (rank == 0 && t == 0) {
                Grid G = {};
                for (int c = 0; c < 3; ++c) G.dim[c] = 1;
                G.b_cut = kRadBins - 1;
                G.pad = total == 0 || !ok;
                *P.grid = G;
                *P.npairs = 0;
                P.cell_start[0] = 0;
                P.cell_start[1] = total;
                if (!ok) atomicOr(P.err, ERR_NONFINITE);
            }
            return;
        }
        if (t < 7) {
            unsigned int m = 0u;
            for (unsigned r = 0; r < ctas; ++r) m = max(m, s_all_kept[r][t]);
            s_kept[t] = m;
        }
        for (int base = 0; base < n; base += bd) {
            const bool in = base + t < n && s_cell[base + t] >= 0;
            const unsigned act = __ballot_sync(0xffffffffu, in);
            if (in) hist_add(s_hist, act, s_sph[base + t].w);
        }
        __syncthreads();
        share_hist();
        cluster_sync();
    }
    {
        const unsigned *bounds = groups ? s_kept : s_bounds;
        float r_cut;
        const int b_cut =
            choose_cut<kRadBins / kGridThreads>(s_hist_all, P.big_cap, 16, ord_dec(bounds[6]), s_hist, &r_cut);
        bool some;
        G = make_grid_from(bounds, P.table, some, r_cut, b_cut, true);
        if (!groups) ok = some;
        if (!ok) G.pad = 1;
    }
    const unsigned int big = big_threshold(G.b_cut);
    const int cells = (int)min((long long)G.dim[0] * G.dim[1] * G.dim[2], (long long)P.table);
    int sh = 5;  // cells per CTA: 2^sh, at most cells_cap (the table holds at most cells_cap x ctas cells)
    while (((int)ctas << sh) < cells) ++sh;
    if (rank == 0 && t == 0) {
        *P.grid = G;
        *P.npairs = 0;
        if (!ok) atomicOr(P.err, ERR_NONFINITE);
    }
    for (int base = 0; base < n; base += 4 * bd) {  // four additions under way per thread
        int cell[4], place[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = base + k * bd + t;
            cell[k] = -1;
            if (i >= n || (groups && s_cell[i] < 0)) continue;
            const float4 sp = s_sph[i];
            if (__float_as_uint(sp.w) > big) {
                const int slot = atomicAdd(P.bp_hist + kRadBins, 1);
                if (slot < P.big_cap) P.big_list[slot] = g0 + i;
                P.spheres[g0 + i] = sp;
            }
            cell[k] = bp_cell(G, sp);
            place[k] = cluster_add(in_cta(s_count + (cell[k] & ((1 << sh) - 1)), cell[k] >> sh), 1);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = base + k * bd + t;
            if (cell[k] < 0) continue;
            s_cell[i] = cell[k];
            s_place[i] = place[k];
        }
    }
    cluster_sync();  // counts complete
    // exclusive scan of this CTA's cells, warp-strided over consecutive cells
    const int lane = t & 31, w = t >> 5, nw = bd >> 5;
    const int own = max(0, min(1 << sh, cells - ((int)rank << sh)));
    const int m = (own + 32 * nw - 1) / (32 * nw), c0 = w * m * 32;
    int sum = 0;
    for (int j = 0; j < m; ++j) {
        const int c = c0 + 32 * j + lane;
        sum += c < own ? s_count[c] : 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) ws[w] = sum;
    __syncthreads();
    if (w == 0) {  // exclusive prefix of the warp totals (at most 16 warps)
        const int a = lane < nw ? ws[lane] : 0;
        const int ia = warp_incl_scan(a);
        __syncwarp();
        if (lane < nw) ws[lane] = ia - a;
        const int total = __shfl_sync(0xffffffffu, ia, 31);
        if (lane < (int)ctas) cluster_store(in_cta(s_tot + rank, lane), (unsigned)total);
    }
    __syncthreads();
    int off = ws[w];
    for (int j = 0; j < m; ++j) {
        const int c = c0 + 32 * j + lane;
        const int v = c < own ? s_count[c] : 0;
        const int iv = warp_incl_scan(v);
        if (c < own) s_count[c] = off + iv - v;
        off += __shfl_sync(0xffffffffu, iv, 31);
    }
    cluster_sync();  // the ranges' starts and totals
    if (t == 0) {  // totals to the ranges' first entries
        int a = 0;
        for (unsigned r = 0; r < ctas; ++r) {
            const int v = s_tot[r];
            s_tot[r] = a;
            a += v;
        }
        if (rank == 0) P.cell_start[cells] = a;
    }
    __syncthreads();
    {
        const int *seg_group = P.seg_group;
        int *cell_pills = P.cell_pills, *cell_grp = P.cell_grp;
        float4 *cell_sph = P.cell_sph;
        for (int base = 0; base < n; base += 4 * bd) {
            int pos[4], grp[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = base + k * bd + t, cell = i < n ? s_cell[i] : -1, r = cell >> sh;
                pos[k] = -1;
                if (cell < 0) continue;
                pos[k] = cluster_load(in_cta(s_count + (cell & ((1 << sh) - 1)), r));
                grp[k] = seg_group[g0 + i];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = base + k * bd + t;
                if (pos[k] < 0) continue;
                const int at = s_tot[s_cell[i] >> sh] + pos[k] + s_place[i];
                cell_pills[at] = g0 + i;
                cell_sph[at] = s_sph[i];
                cell_grp[at] = grp[k];
            }
        }
    }
    {
        int *cell_start = P.cell_start;
        const int base = s_tot[rank], first = (int)rank << sh;
        for (int c = t; c < own; c += bd) cell_start[first + c] = base + s_count[c];
    }
    cluster_sync();  // the others have read this CTA's starts
}

// First sweep of a substep with the previous substep's velocity update and
// this substep's prediction folded in (see rod_item_first).
__global__ void __launch_bounds__(256) batch_rod_first_kernel(BatchArgs A, int finish_prev, float tau)
{
    __shared__ BatchScene sb;
    extern __shared__ float4 smem[];
    int local, nblk;
    batch_enter(A, K_ROD, sb, local, nblk);
    rod_item_first(sb.P, local, finish_prev != 0, tau, sb.pills != 0, smem);
}

// Whether a scene's contact passes read world and pill packs (Params::XW, PB):
// from the second sweep of a substep on, when the pair search found at least
// two pairs per pill.  The sweep before such a pass writes them (48 bytes a
// vertex); the same decision on both sides, from the pair count of the substep.
// A multi-scene frame without packs, with this rule and with packs always, in us: settled
// strands, 13,000 pills (11 pairs a pill) 1,354, 1,324, 1,328, and 26,000 2,908, 2,680,
// 2,670; falling, 26,000 pills (4) 1,102, 1,073, 1,068; 30 rigs of 40 muscles (next to
// none) 1,902, 1,907, 1,922.
constexpr int kPackPairs = 2;
__device__ __forceinline__ bool packs_used(const Params &P, bool first_sweep)
{
    return !first_sweep && P.XW && *P.npairs >= kPackPairs * P.ns;
}

// One colour sweep of every work item (contact path).
__global__ void __launch_bounds__(256, 2) batch_rod_kernel(BatchArgs A, int first, int apply)
{
    __shared__ BatchScene sb;
    extern __shared__ float4 smem[];
    int local, nblk;
    batch_scene(A, K_ROD, sb, local, nblk);
    RodStage S;
    rod_stage_rest(sb.P, local, first != 0, S);
    // after a contact pass: the state and the pair count are those it started from
    if (!first) rod_stage_state(sb.P, S, smem);
    // read after rod_run's first barrier
    if (threadIdx.x == 0 && !packs_used(sb.P, first != 0)) sb.P.XW = nullptr;
    pdl_wait();
    pdl_trigger();
    if (first) rod_stage_state(sb.P, S, smem);
    rod_run(sb.P, S, apply != 0, smem);
}

// Every substep of the frame (no contacts).
__global__ void __launch_bounds__(256, 2) batch_rod_frame_kernel(BatchArgs A, int substeps, int n_iter)
{
    __shared__ BatchScene sb;
    extern __shared__ float4 smem[];
    int local, nblk;
    batch_enter(A, K_ROD, sb, local, nblk);
    rod_frame_item(sb.P, local, substeps, n_iter, smem);
}

// Jacobi contact pass (Sec. 7.2) after the sweep `first`: pairs, then half-plane
// vertices, over the scene's CTAs.
__global__ void __launch_bounds__(kElemThreads, 4) batch_contact_kernel(BatchArgs A, int first)
{
    __shared__ BatchScene sb;
    __shared__ QueuedPair queue[kElemThreads / 32][64];
    int local, nblk;
    batch_scene(A, K_CONTACT, sb, local, nblk);
    Params &P = sb.P;
    if (first) pdl_wait();  // the pair search is finished before any later pass's sweep begins
    const int np_all = sb.pills ? *P.npairs : 0;
    if (threadIdx.x == 0 && !packs_used(P, first != 0)) {
        P.XW = nullptr;
        P.PB = nullptr;
    }
    if (!first) pdl_wait();
    __syncthreads();
    const int np = min(np_all, P.max_pairs);
    if (local == 0 && threadIdx.x == 0 && np_all > P.max_pairs) atomicOr(P.err, ERR_OVERFLOW);
    const int nvp = P.n_planes > 0 ? P.nv : 0;
    const float at = P.contact_alpha * P.inv_h2;
    const int threads = nblk * blockDim.x;
    const int lane = threadIdx.x & 31, warp = (local * blockDim.x + threadIdx.x) >> 5;
    if (!P.contact_threads && (long long)np * 16 <= threads) {
        // few pairs (an animated scene's usual case, a few per cent of its pills): a
        // warp per pair, at most two pairs per warp, the search's steps four at a
        // time (three rounds against ten steps)
        pdl_trigger();
        for (int i = warp; i < np; i += threads >> 5) contact_pair_warp(P, i, at, lane);
    } else {
        // a thread per pair, the pairs that may touch compacted per warp; the next sweep is
        // let in after them, not beside them (2,000 settled strands 1.46 -> 1.39 ms a frame)
        contact_pairs_compacted(P, np, at, warp, threads >> 5, queue[threadIdx.x >> 5], lane);
        pdl_trigger();
    }
    for (int i = local * blockDim.x + threadIdx.x; i < nvp; i += threads) contact_planes(P, i, at);
}

// Bundle shape matching after the substep's last contact pass (see
// match_cross_section), one warp per cross-section.
__global__ void __launch_bounds__(kElemThreads) batch_bundle_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_BUNDLE, sb, local, nblk);
    const int warps = kElemThreads / 32;
    for (int c = local * warps + (threadIdx.x >> 5); c < sb.P.n_xs; c += nblk * warps) match_cross_section(sb.P, c);
}

// The start of a substep without its first sweep (the sweep runs beside the
// broadphase): the previous substep's velocity update (`finish_prev`) and the
// prediction of every vertex and segment.
__global__ void __launch_bounds__(kElemThreads) batch_advance_kernel(BatchArgs A, int finish_prev, float tau)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_scene(A, K_ELEM, sb, local, nblk);
    const Params &P = sb.P;
    const int i = local * blockDim.x + threadIdx.x, nv = P.nv;
    const bool fin = finish_prev != 0, vertex = i < nv, segment = !vertex && i < nv + P.ns, world = sb.pills != 0;
    // loaded while the previous substep's last contact pass still runs, unless shape
    // matching or the warm start runs in between
    const bool state = fin && P.n_xs == 0;
    AdvanceVertex V;
    AdvanceSegment G;
    if (vertex) advance_vertex_load(P, i, fin, state, tau, world, V);
    if (segment) advance_segment_load(P, i - nv, fin, state, G);
    pdl_wait();
    pdl_trigger();
    if (sb.pills && local == 0 && threadIdx.x < 8) P.bounds[threadIdx.x] = 0u;
    if (vertex) advance_vertex_at(P, i, fin, state, world, V);
    if (segment) advance_segment_at(P, i - nv, fin, state, G);
}

// Warm start from the bones before the frame's first substep (scenes with a warm-start table).
__global__ void __launch_bounds__(kElemThreads) batch_warm_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_WARM, sb, local, nblk);
    const Params &P = sb.P;
    const int v = local * blockDim.x + threadIdx.x;
    if (v < P.nv) P.X[v] = warm_vertex(P, v, P.X[v]);
}

// Velocity update after the last contact pass.
__global__ void __launch_bounds__(kElemThreads) batch_finish_kernel(BatchArgs A, int apply)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_ELEM, sb, local, nblk);
    const Params &P = sb.P;
    const int i = local * blockDim.x + threadIdx.x;
    if (i < P.nv)
        finish_vertex_at(P, i, apply != 0);
    else if (i < P.nv + P.ns)
        finish_segment_at(P, i - P.nv);
}

// ---------------------------------------------------------------- end of frame
// Skinning frames (scenes with a mesh), the bone pose handed on (previous :=
// target, and the frame's target kept as the scene's own), and the error word
// mirrored to the host.
__global__ void __launch_bounds__(kElemThreads) batch_end_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_END, sb, local, nblk);
    const Params &P = sb.P;
    const int g = local * blockDim.x + threadIdx.x;
    if (sb.n_mesh > 0 && g < P.ns) lbs_frame_at(P, sb.LQ, sb.LC, sb.sperm, sb.frames, g);
    if (local == 0) {
        for (int b = threadIdx.x; b < sb.n_bones; b += blockDim.x) {
            const float4 q = P.bq1[b];
            const float t0 = P.bt1[3 * b], t1 = P.bt1[3 * b + 1], t2 = P.bt1[3 * b + 2];
            sb.bq0[b] = q;
            sb.bt0[3 * b] = t0;
            sb.bt0[3 * b + 1] = t1;
            sb.bt0[3 * b + 2] = t2;
            if (P.bq1 != sb.bq1_own) {
                sb.bq1_own[b] = q;
                sb.bt1_own[3 * b] = t0;
                sb.bt1_own[3 * b + 1] = t1;
                sb.bt1_own[3 * b + 2] = t2;
            }
        }
        if (threadIdx.x == 0) *(volatile int *)sb.herr = *(volatile int *)P.err;
    }
}

__global__ void __launch_bounds__(kElemThreads) batch_skin_kernel(BatchArgs A)
{
    __shared__ BatchScene sb;
    int local, nblk;
    batch_enter(A, K_MESH, sb, local, nblk);
    const int span = blockDim.x * kLbsBatch;
    for (int base = local * span; base < sb.n_mesh; base += nblk * span)
        lbs_vertices(base + threadIdx.x, blockDim.x, sb.n_mesh, sb.P.ns, sb.rest, sb.idx, sb.w, sb.frames, sb.out,
                     sb.P.err);
}

// ---------------------------------------------------------------- host side
namespace {

// launch_dependent in thread-block clusters of `ctas`.
template <typename... KArgs, typename... Args>
void launch_clusters(void (*kernel)(KArgs...), int grid, int ctas, int block, int smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = ctas;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

// CTAs of the cluster that builds a scene's grid: eight where that fills no more
// than the GPU's two CTAs per SM, fewer for many scenes, but enough for the
// largest scene's cells and pills (kGridCellsMax, kGridSliceMax per CTA).
int grid_cluster(int scenes, int max_ns, int max_table)
{
    int c = scenes * kGridClusterMax <= 2 * device_sm_count() ? kGridClusterMax : scenes <= device_sm_count() ? 4 : 2;
    while (c < kGridClusterMax && (max_table > c * kGridCellsMax || max_ns > c * kGridSliceMax)) c *= 2;
    return c;
}

// CTAs for a scene's `part` of the group's `all` pills: what it could use, `want`,
// within its share of the four CTAs an SM holds.  A CTA without work still costs its
// start: 64 scenes with 1,738 CTAs each for the search and the passes, most of
// them idle, took 3.00 ms a frame, with 577 2.86.
int resident_share(int want, int part, long long all)
{
    const long long most = 4LL * device_sm_count() * part / std::max(all, 1LL);
    return (int)std::max(1LL, std::min((long long)want, most));
}

// Groups of few pills do not fill the GPU with a thread per pill: several lanes
// search a pill's neighbours, and a contact CTA covers fewer pills.  With one, two,
// four and eight lanes, in us: 200 muscles, 6,910 pills, two frames 1,014, 977, 967,
// 961 (few pills stay after the cull); a frame of settled strands, 14,300 pills, 1,512,
// 1,330, 1,290, 1,276, and 19,500 1,788, 1,583, 1,552, 1,532; of falling ones, 9,100
// pills, 719, 688, 672, 676, and 19,500 878, 826, 832, 834.
constexpr int kSmallGroup = 20000, kEmitLanesSmall = 4, kContactPillsSmall = 64;
constexpr int kMeshPerThread = 16;  // kLbsBatch vertices per round, 16 / kLbsBatch rounds

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }
int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

}  // namespace

}  // namespace viper

struct viper_batch {
    struct Stage {
        char *h = nullptr;  // pinned
        char *d = nullptr;  // device
        size_t cap = 0;
        cudaEvent_t done = nullptr;  // the last call that used this stage has finished on the device
        bool used = false;
    };
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    Stage stage[2];
    int cur = 0;
    std::vector<cudaEvent_t> ev;  // ordering after the scenes' streams
    cudaEvent_t ev_after = nullptr;
    cudaStream_t side = nullptr;  // the branch of a sequence with the first sweep
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    long long launches = 0;
};

namespace viper {
namespace {

int stage_reserve(viper_batch::Stage &S, size_t bytes)
{
    if (S.used && cudaEventSynchronize(S.done) != cudaSuccess) return VIPER_ECUDA;
    if (S.cap >= bytes) return VIPER_OK;
    size_t cap = std::max(bytes, 2 * S.cap);
    if (S.h) cudaFreeHost(S.h);
    if (S.d) cudaFree(S.d);
    S.h = nullptr;
    S.d = nullptr;
    S.cap = 0;
    if (cudaHostAlloc((void **)&S.h, cap, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        S.h = nullptr;
        return VIPER_ENOMEM;
    }
    if (cudaMalloc((void **)&S.d, cap) != cudaSuccess) {
        cudaGetLastError();
        cudaFreeHost(S.h);
        S.h = nullptr;
        S.d = nullptr;
        return VIPER_ENOMEM;
    }
    S.cap = cap;
    return VIPER_OK;
}

// A second stream and two events for the branch of a sequence with the first sweep.
struct Fork {
    cudaStream_t side;
    cudaEvent_t ev_fork, ev_join;
};

// Launch shape of one sequence: blocks per kernel kind over all its scenes.
struct Shape {
    int tot[K_KINDS] = {};
    bool small = false;        // few pills (kSmallGroup)
    long long all_pills = 0;   // segments of the group's scenes
    int threads = 0, smem = 16;
    bool cp = false, fused_grid = true;
    int cluster = kGridClusterMax, cells_cap = 32, slice_cap = 32, groups_cap = 0;  // grid build: CTAs per scene, shared memory
};

// Device view of one scene for a frame of sub-step h (b.P.bq1 / bt1: the
// scene's own target pose; the caller may point them elsewhere), and its
// blocks per kernel kind.
void fill_scene(BatchScene &b, int cnt[K_KINDS], viper_scene *s, const viper_batch_item &it, double h, bool cp,
                const Shape &sh)
{
    memset(&b, 0, sizeof(b));
    b.P = s->P;
    if ((s->flags & VIPER_FLAG_CONTACTS) && cp) {
        b.P.XW = s->xw;
        b.P.PB = s->pb;
    }
    b.P.h = (float)h;
    b.P.inv_h = (float)(1.0 / h);
    b.P.inv_h2 = (float)(1.0 / (h * h));
    b.LQ = s->LQ;
    b.LC = s->LC;
    b.sperm = s->d_sperm;
    b.frames = s->frames;
    b.rest = reinterpret_cast<const float4 *>(it.rest4);
    b.idx = reinterpret_cast<const int4 *>(it.idx4);
    b.w = reinterpret_cast<const float4 *>(it.w4);
    b.out = reinterpret_cast<float4 *>(it.out4);
    b.n_mesh = it.n_mesh;
    b.bq0 = const_cast<float4 *>(s->P.bq0);
    b.bq1_own = const_cast<float4 *>(s->P.bq1);
    b.bt0 = const_cast<float *>(s->P.bt0);
    b.bt1_own = const_cast<float *>(s->P.bt1);
    b.herr = s->d_herr;
    b.n_bones = s->n_bones;
    b.pills = (s->flags & VIPER_FLAG_CONTACTS) ? 1 : 0;
    const int nv = s->nv, ns = s->ns;
    cnt[K_ELEM] = cdiv(nv + ns, kElemThreads);
    cnt[K_PILL] = b.pills ? cdiv(ns, kElemThreads) : 0;
    // pair search and contact pass: grid-stride over the scene's pills and pairs, so no
    // more CTAs than stay resident, shared out by size (see resident_share)
    const long long want_emit = (long long)ns * (sh.small ? kEmitLanesSmall : 1);
    cnt[K_EMIT] = b.pills ? resident_share(cdiv(want_emit, 32 * kEmitWarpsB), ns, sh.all_pills) : 0;
    cnt[K_SCAN] = b.pills ? 1 : 0;
    cnt[K_GRID] = b.pills ? sh.cluster : 0;
    cnt[K_ROD] = s->n_items;
    const int touch = ns + (s->n_planes > 0 ? nv : 0);
    cnt[K_CONTACT] =
        cp ? resident_share(cdiv(touch, sh.small ? kContactPillsSmall : kElemThreads), ns, sh.all_pills) : 0;
    cnt[K_END] = it.n_mesh > 0 ? std::max(1, cdiv(ns, kElemThreads)) : 1;
    cnt[K_MESH] = cdiv(it.n_mesh, kElemThreads * kMeshPerThread);
    cnt[K_BUNDLE] = cp ? cdiv(s->P.n_xs, kElemThreads / 32) : 0;
    cnt[K_WARM] = s->P.warm ? cdiv(nv, kElemThreads) : 0;
}

void shape_add(Shape &sh, const viper_scene *s, bool cp)
{
    sh.cp = cp;
    sh.smem = std::max(sh.smem, cp ? s->smem_iter : s->smem_full);
    if (cp && (s->flags & VIPER_FLAG_CONTACTS)) {
        if (s->ns > kGridMaxPills) sh.fused_grid = false;
        sh.cells_cap = std::max(sh.cells_cap, s->P.table / sh.cluster);
        sh.slice_cap = std::max(sh.slice_cap, cdiv(s->ns, 4 * sh.cluster) * 4);
        if (s->P.n_groups <= kGridGroupsMax) sh.groups_cap = std::max(sh.groups_cap, s->P.n_groups);
    }
    sh.threads = s->block_threads;
}

// Enqueue the frame's launch sequence on st; returns the number of kernels or
// -1.  With `prof`, each launch is bracketed by that scene's profiling events.
long long enqueue_sequence(const BatchArgs &A, const Shape &sh, int substeps, int iterations, cudaStream_t st,
                           viper_scene *prof, const Fork *fork)
{
    const int *tot = sh.tot;
    const int threads = sh.threads, smem = sh.smem;
    const bool cp = sh.cp, fused_grid = sh.fused_grid;
    const void *rod_fn = cp ? reinterpret_cast<const void *>(batch_rod_kernel)
                            : reinterpret_cast<const void *>(batch_rod_frame_kernel);
    if (raise_smem_limit(rod_fn, smem) != 0) return -1;
    if (cp && raise_smem_limit(reinterpret_cast<const void *>(batch_rod_first_kernel), smem) != 0) return -1;
    const int grid_smem = grid_smem_bytes(sh.cells_cap, sh.slice_cap, sh.groups_cap);
    if (tot[K_GRID] > 0 && fused_grid &&
        raise_smem_limit(reinterpret_cast<const void *>(batch_grid_kernel), grid_smem) != 0)
        return -1;
    long long L = 0;
    auto go = [&](int cls, auto &&fn) {
        ProfScope ps(prof, cls);
        fn();
        ++L;
    };
    auto broadphase = [&](cudaStream_t bs) {
        if (tot[K_PILL] <= 0) return;
        if (fused_grid) {
            go(PROF_BROADPHASE, [&] {
                launch_clusters(batch_grid_kernel, tot[K_GRID], sh.cluster, kGridThreads, grid_smem, bs, A, sh.cells_cap,
                                sh.slice_cap, sh.groups_cap);
            });
        } else {
            go(PROF_BROADPHASE, [&] { launch_dependent(batch_bounds_kernel, tot[K_PILL], kElemThreads, 0, bs, A); });
            go(PROF_BROADPHASE, [&] { launch_dependent(batch_count_kernel, tot[K_PILL], kElemThreads, 0, bs, A); });
            go(PROF_BROADPHASE, [&] { launch_dependent(batch_scan_kernel, tot[K_SCAN], kScanThreadsB, 0, bs, A); });
            go(PROF_BROADPHASE, [&] { launch_dependent(batch_scatter_kernel, tot[K_PILL], kElemThreads, 0, bs, A); });
        }
        go(PROF_PAIRS, [&] {
            launch_dependent(sh.small ? batch_emit_kernel<kEmitLanesSmall> : batch_emit_kernel<1>, tot[K_EMIT], 32 * kEmitWarpsB, 0, bs, A);
        });
    };
    // the first sweep on a second branch beside the broadphase (not while profiling:
    // the per-class events bracket one stream)
    const bool forked = fork && fork->side && tot[K_PILL] > 0 && (!prof || prof->prof_class == PROF_NONE);
    auto contact = [&](int first) {
        go(PROF_CONTACT, [&] { launch_dependent(batch_contact_kernel, tot[K_CONTACT], kElemThreads, 0, st, A, first); });
    };
    if (tot[K_WARM] > 0) go(PROF_ELEM, [&] { launch_dependent(batch_warm_kernel, tot[K_WARM], kElemThreads, 0, st, A); });
    if (cp && iterations > 0) {
        // per substep: [finish + predict + sweep 0] | grid | emit | contact | {sweep | contact} x (I - 1)
        for (int k = 0; k < substeps; ++k) {
            const float tau = (float)((double)(k + 1) / substeps);  // as the one-scene path
            if (forked) {
                // advance | [grid, pair search] beside [first sweep] | contact ...; the grid and
                // the pair search take longer than the sweep, so they follow on the main
                // stream, where their prologues overlap what is before them
                go(PROF_ELEM, [&] { launch_dependent(batch_advance_kernel, tot[K_ELEM], kElemThreads, 0, st, A, k > 0 ? 1 : 0, tau); });
                if (cudaEventRecord(fork->ev_fork, st) != cudaSuccess ||
                    cudaStreamWaitEvent(fork->side, fork->ev_fork, 0) != cudaSuccess)
                    return -1;
                broadphase(st);
                go(PROF_ROD, [&] { launch_dependent(batch_rod_kernel, tot[K_ROD], threads, smem, fork->side, A, 1, 0); });
                if (cudaEventRecord(fork->ev_join, fork->side) != cudaSuccess ||
                    cudaStreamWaitEvent(st, fork->ev_join, 0) != cudaSuccess)
                    return -1;
            } else {
                go(PROF_ROD, [&] { launch_dependent(batch_rod_first_kernel, tot[K_ROD], threads, smem, st, A, k > 0 ? 1 : 0, tau); });
                broadphase(st);
            }
            contact(1);
            for (int i = 1; i < iterations; ++i) {
                go(PROF_ROD, [&] { launch_dependent(batch_rod_kernel, tot[K_ROD], threads, smem, st, A, 0, 1); });
                contact(0);
            }
            if (tot[K_BUNDLE] > 0)
                go(PROF_ELEM, [&] { launch_dependent(batch_bundle_kernel, tot[K_BUNDLE], kElemThreads, 0, st, A); });
        }
        go(PROF_ELEM, [&] { launch_dependent(batch_finish_kernel, tot[K_ELEM], kElemThreads, 0, st, A, 1); });
    } else if (!cp) {
        go(PROF_ROD, [&] { launch_dependent(batch_rod_frame_kernel, tot[K_ROD], threads, smem, st, A, substeps, iterations); });
    } else {
        // contact path without iterations: prediction, broadphase, velocity update
        for (int k = 0; k < substeps; ++k) {
            const float tau = (float)((double)(k + 1) / substeps);  // as the one-scene path
            go(PROF_ELEM, [&] { launch_dependent(batch_predict_kernel, tot[K_ELEM], kElemThreads, 0, st, A, tau); });
            broadphase(st);
            go(PROF_ELEM, [&] { launch_dependent(batch_finish_kernel, tot[K_ELEM], kElemThreads, 0, st, A, 0); });
        }
    }
    go(PROF_ELEM, [&] { launch_dependent(batch_end_kernel, tot[K_END], kElemThreads, 0, st, A); });
    if (tot[K_MESH] > 0) go(PROF_LBS, [&] { launch_dependent(batch_skin_kernel, tot[K_MESH], kElemThreads, 0, st, A); });
    return cudaGetLastError() == cudaSuccess ? L : -1;
}

// One launch sequence for the scenes idx (same CTA size; contact path or not).
int run_group(viper_batch *B, const viper_batch_item *items, const std::vector<int> &idx, float dt, int substeps,
              int iterations, bool cp)
{
    const int n = (int)idx.size();
    size_t nb_total = 0;
    for (int i : idx)
        if (items[i].bone_quat) nb_total += (size_t)items[i].scene->n_bones;
    const size_t o_off = align16(sizeof(BatchScene) * n);
    const size_t o_bq = align16(o_off + sizeof(int) * K_KINDS * (size_t)(n + 1));
    const size_t o_bt = o_bq + sizeof(float4) * nb_total;
    const size_t bytes = o_bt + sizeof(float) * 3 * nb_total;
    viper_batch::Stage &S = B->stage[B->cur];
    B->cur ^= 1;
    int rc = stage_reserve(S, bytes);
    if (rc) return rc;

    BatchScene *hs = reinterpret_cast<BatchScene *>(S.h);
    int *off = reinterpret_cast<int *>(S.h + o_off);
    float4 *hbq = reinterpret_cast<float4 *>(S.h + o_bq);
    float *hbt = reinterpret_cast<float *>(S.h + o_bt);
    const float4 *dbq = reinterpret_cast<const float4 *>(S.d + o_bq);
    const float *dbt = reinterpret_cast<const float *>(S.d + o_bt);
    const double h = (double)dt / substeps;
    size_t bcur = 0;
    Shape sh;
    long long group_pills = 0;
    int pill_scenes = 0, max_ns = 0, max_table = 0;
    for (int i : idx)
        if (items[i].scene->flags & VIPER_FLAG_CONTACTS) {
            const viper_scene *s = items[i].scene;
            group_pills += s->ns;
            ++pill_scenes;
            max_ns = std::max(max_ns, s->ns);
            max_table = std::max(max_table, s->P.table);
        }
    sh.cluster = grid_cluster(pill_scenes, max_ns, max_table);
    sh.small = group_pills <= kSmallGroup;
    for (int i : idx) sh.all_pills += items[i].scene->ns;
    for (int c = 0; c < K_KINDS; ++c) off[c * (n + 1)] = 0;
    for (int k = 0; k < n; ++k) {
        const viper_batch_item &it = items[idx[k]];
        viper_scene *s = it.scene;
        BatchScene &b = hs[k];
        int cnt[K_KINDS];
        fill_scene(b, cnt, s, it, h, cp, sh);
        if (it.bone_quat && s->n_bones > 0) {  // this frame's target pose, from the call's table
            memcpy(hbq + bcur, it.bone_quat, sizeof(float4) * s->n_bones);
            memcpy(hbt + 3 * bcur, it.bone_trans, sizeof(float) * 3 * s->n_bones);
            b.P.bq1 = dbq + bcur;
            b.P.bt1 = dbt + 3 * bcur;
            bcur += (size_t)s->n_bones;
        }
        for (int c = 0; c < K_KINDS; ++c) off[c * (n + 1) + k + 1] = off[c * (n + 1) + k] + cnt[c];
        shape_add(sh, s, cp);
    }
    for (int c = 0; c < K_KINDS; ++c) sh.tot[c] = off[c * (n + 1) + n];
    // a warp per contact pair shortens one scene's chain but multiplies the
    // lanes' work; once the scenes' contact passes fill the GPU, throughput
    // decides: one thread per pair
    if (!sh.small && sh.tot[K_CONTACT] > device_sm_count())
        for (int k = 0; k < n; ++k) hs[k].P.contact_threads = 1;

    cudaStream_t st = B->stream;
    if (cudaMemcpyAsync(S.d, S.h, bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return VIPER_ECUDA;
    BatchArgs A{reinterpret_cast<const BatchScene *>(S.d), reinterpret_cast<const int *>(S.d + o_off), n};
    const Fork fk{B->side, B->ev_fork, B->ev_join};
    const long long L = enqueue_sequence(A, sh, substeps, iterations, st, nullptr, &fk);
    if (L < 0) return VIPER_ECUDA;
    B->launches += L;
    if (cudaEventRecord(S.done, st) != cudaSuccess) return VIPER_ECUDA;
    S.used = true;
    return VIPER_OK;
}

}  // namespace

// A larger scene alone runs the multi-kernel path: packs from the first sweep on and
// passes over the whole GPU, but no cull.  The line is where rigs cross, which the cull
// helps most (two frames, here and there, in us: 500 muscles, 18,061 pills, 1,515 and
// 1,775; 620, 22,177 pills, 1,865 and 1,825; 190 bundles, 19,950 pills, 1,050 and 1,240;
// 350, 36,750 pills, 1,295 and 1,373).  Strands cross at half of it (a frame, settled:
// 10,400 pills 1,091 and 1,084, 19,500 1,514 and 1,428, 26,000 2,578 and 1,664; falling:
// 7,150 pills 651 and 708, 19,500 829 and 739, 26,000 992 and 790).
constexpr int kSelfMaxPills = 20000;

bool self_batch_ok(const viper_scene *s)
{
    return s->resident_nv == s->nv && s->n_items > 0 &&
           (!(s->flags & VIPER_FLAG_CONTACTS) || s->ns <= kSelfMaxPills);
}

int self_batch_capture(viper_scene *s, float dt, int substeps, int iterations, cudaGraph_t *graph,
                       long long *launches)
{
    const size_t o_off = align16(sizeof(BatchScene));
    const size_t bytes = o_off + sizeof(int) * K_KINDS * 2;
    if (!s->self_table) {
        int rc = scene_alloc(s, bytes, &s->self_table);
        if (rc) return rc;
    }
    std::vector<char> h(bytes, 0);
    BatchScene *b = reinterpret_cast<BatchScene *>(h.data());
    int *off = reinterpret_cast<int *>(h.data() + o_off);
    viper_batch_item it;
    memset(&it, 0, sizeof(it));
    it.scene = s;
    const bool cp = scene_contact_path(s);
    int cnt[K_KINDS];
    Shape sh;
    sh.small = s->ns <= kSmallGroup;
    sh.all_pills = s->ns;
    sh.cluster = grid_cluster(1, s->ns, s->P.table);
    fill_scene(*b, cnt, s, it, (double)dt / substeps, cp, sh);  // bones: the scene's own target pose
    shape_add(sh, s, cp);
    for (int c = 0; c < K_KINDS; ++c) {
        off[2 * c] = 0;
        off[2 * c + 1] = cnt[c];
        sh.tot[c] = cnt[c];
    }
    // stream-ordered after any replay of an earlier graph that reads the table
    if (cudaMemcpyAsync(s->self_table, h.data(), bytes, cudaMemcpyHostToDevice, s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
        return VIPER_ECUDA;
    const char *t = static_cast<const char *>(s->self_table);
    BatchArgs A{reinterpret_cast<const BatchScene *>(t), reinterpret_cast<const int *>(t + o_off), 1};
    s->prof_used = 0;
    if (cudaStreamBeginCapture(s->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return VIPER_ECUDA;
    const Fork fk{s->side, s->ev_fork, s->ev_join};
    const long long L = enqueue_sequence(A, sh, substeps, iterations, s->stream, s, &fk);
    cudaError_t ce = cudaStreamEndCapture(s->stream, graph);
    if (L < 0 || ce != cudaSuccess) {
        if (ce == cudaSuccess && *graph) cudaGraphDestroy(*graph);
        *graph = nullptr;
        return VIPER_ECUDA;
    }
    *launches = L;
    return VIPER_OK;
}

}  // namespace viper

using namespace viper;

extern "C" {

int viper_batch_create(void *stream, viper_batch **out)
{
    if (!out) return VIPER_EINVAL;
    viper_batch *B = new viper_batch();
    bool ok = true;
    if (stream) {
        B->stream = (cudaStream_t)stream;
    } else {
        ok = cudaStreamCreateWithFlags(&B->stream, cudaStreamNonBlocking) == cudaSuccess;
        B->own_stream = ok;
    }
    for (int i = 0; i < 2 && ok; ++i)
        ok = cudaEventCreateWithFlags(&B->stage[i].done, cudaEventDisableTiming) == cudaSuccess;
    if (ok) ok = cudaEventCreateWithFlags(&B->ev_after, cudaEventDisableTiming) == cudaSuccess;
    if (ok) ok = cudaStreamCreateWithFlags(&B->side, cudaStreamNonBlocking) == cudaSuccess;
    if (ok) ok = cudaEventCreateWithFlags(&B->ev_fork, cudaEventDisableTiming) == cudaSuccess;
    if (ok) ok = cudaEventCreateWithFlags(&B->ev_join, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
        viper_batch_destroy(B);
        return VIPER_ECUDA;
    }
    *out = B;
    return VIPER_OK;
}

void viper_batch_destroy(viper_batch *B)
{
    if (!B) return;
    if (B->stream) cudaStreamSynchronize(B->stream);
    for (auto &S : B->stage) {
        if (S.h) cudaFreeHost(S.h);
        if (S.d) cudaFree(S.d);
        if (S.done) cudaEventDestroy(S.done);
    }
    for (cudaEvent_t e : B->ev) cudaEventDestroy(e);
    if (B->ev_after) cudaEventDestroy(B->ev_after);
    if (B->side) {
        cudaStreamSynchronize(B->side);
        cudaStreamDestroy(B->side);
    }
    if (B->ev_fork) cudaEventDestroy(B->ev_fork);
    if (B->ev_join) cudaEventDestroy(B->ev_join);
    if (B->own_stream) cudaStreamDestroy(B->stream);
    delete B;
}

void *viper_batch_stream(const viper_batch *B) { return B ? (void *)B->stream : nullptr; }

long long viper_batch_launch_count(const viper_batch *B) { return B ? B->launches : 0; }

int viper_batch_step(viper_batch *B, const viper_batch_item *items, int n, float dt, int substeps, int iterations,
                     int *status)
{
    if (!B || n < 0 || (n > 0 && !items) || !(dt > 0) || substeps <= 0 || iterations < 0) return VIPER_EINVAL;
    std::vector<viper_scene *> seen(n);
    for (int i = 0; i < n; ++i) {
        const viper_batch_item &it = items[i];
        if (!it.scene || (!it.bone_quat) != (!it.bone_trans) || it.n_mesh < 0) return VIPER_EINVAL;
        if (it.n_mesh > 0 && (!it.rest4 || !it.idx4 || !it.w4 || !it.out4)) return VIPER_EINVAL;
        if (it.n_mesh > 0 && ((reinterpret_cast<uintptr_t>(it.rest4) | reinterpret_cast<uintptr_t>(it.idx4) |
                               reinterpret_cast<uintptr_t>(it.w4) | reinterpret_cast<uintptr_t>(it.out4)) & 15u))
            return VIPER_EINVAL;  // float4 / int4 arrays
        seen[i] = it.scene;
    }
    std::sort(seen.begin(), seen.end());
    if (std::adjacent_find(seen.begin(), seen.end()) != seen.end()) return VIPER_EINVAL;

    // latched errors; groups of scenes that share one launch sequence
    std::vector<int> st(n, VIPER_OK), single;
    std::map<std::pair<int, int>, std::vector<int>> groups;  // (contact path, CTA size) -> items
    for (int i = 0; i < n; ++i) {
        viper_scene *s = items[i].scene;
        st[i] = scene_poll_latched(s);
        if (st[i] == VIPER_ENONFINITE) continue;
        if (s->resident_nv == s->nv && s->n_items > 0 && !s->P.vvec)
            groups[{scene_contact_path(s) ? 1 : 0, s->block_threads}].push_back(i);
        else
            single.push_back(i);
    }
    // the batch stream runs after work already queued on the scenes' streams
    if ((int)B->ev.size() < n) {
        for (int i = (int)B->ev.size(); i < n; ++i) {
            cudaEvent_t e;
            if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return VIPER_ECUDA;
            B->ev.push_back(e);
        }
    }
    for (auto &g : groups)
        for (int i : g.second) {
            viper_scene *s = items[i].scene;
            if (s->stream == B->stream) continue;
            if (cudaEventRecord(B->ev[i], s->stream) != cudaSuccess) return VIPER_ECUDA;
            if (cudaStreamWaitEvent(B->stream, B->ev[i], 0) != cudaSuccess) return VIPER_ECUDA;
        }
    for (auto &g : groups) {
        int rc = run_group(B, items, g.second, dt, substeps, iterations, g.first.first != 0);
        if (rc) return rc;
    }
    if (!groups.empty()) {
        if (cudaEventRecord(B->ev_after, B->stream) != cudaSuccess) return VIPER_ECUDA;
        for (auto &g : groups)
            for (int i : g.second) {
                viper_scene *s = items[i].scene;
                if (s->stream != B->stream && cudaStreamWaitEvent(s->stream, B->ev_after, 0) != cudaSuccess)
                    return VIPER_ECUDA;
            }
    }
    // scenes outside the shared-memory kernels: one by one on their own streams
    for (int i : single) {
        const viper_batch_item &it = items[i];
        viper_scene *s = it.scene;
        int rc = VIPER_OK;
        if (it.bone_quat && s->n_bones > 0) rc = viper_set_bones(s, s->n_bones, it.bone_quat, it.bone_trans);
        if (rc == VIPER_OK) rc = viper_step(s, dt, substeps, iterations);
        if ((rc == VIPER_OK || rc == VIPER_EOVERFLOW) && it.n_mesh > 0)
            rc = viper_skin(s, it.n_mesh, it.rest4, it.idx4, it.w4, it.out4);
        if (rc != VIPER_OK && rc != VIPER_EOVERFLOW) st[i] = rc;
    }
    if (status)
        for (int i = 0; i < n; ++i) status[i] = st[i];
    return cudaGetLastError() == cudaSuccess ? VIPER_OK : VIPER_ECUDA;
}

}  // extern "C"
