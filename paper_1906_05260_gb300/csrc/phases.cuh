// phases.cuh -- per-element phases of the VIPER solver shared by the
// launch-per-phase kernels (rod.cu, contact.cu) and the persistent frame
// kernel (frame.cu): prediction with kinematic pins, velocity update, contact
// accumulation, broadphase grid helpers, warp and block scans.
#pragma once
#include <mutex>

#include "viper_device.cuh"
#include "viper_impl.h"

namespace viper {

// The dynamic shared-memory limit is a process-wide attribute of a kernel on
// the current device: scenes only ever raise it (under a lock), so a scene
// created later with smaller work items cannot lower it below what an
// earlier scene launches with.
inline int raise_smem_limit(const void *fn, int bytes)
{
    static std::mutex mu;
    struct Entry {
        const void *fn;
        int dev, bytes;
    };
    static Entry seen[64];
    static int n_seen = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    std::lock_guard<std::mutex> lk(mu);
    for (int i = 0; i < n_seen; ++i)
        if (seen[i].fn == fn && seen[i].dev == dev) {
            if (bytes <= seen[i].bytes) return 0;
            if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
                cudaGetLastError();
                return -1;
            }
            seen[i].bytes = bytes;
            return 0;
        }
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    if (n_seen < 64) seen[n_seen++] = Entry{fn, dev, bytes};
    return 0;
}

// Programmatic dependent launch (sm_90 and later): a kernel launched with the
// programmatic stream serialisation attribute may be scheduled while its
// predecessor in the stream still runs.  pdl_wait blocks until the
// predecessor grid has completed and its memory is visible (a no-op for a
// normal launch); pdl_trigger lets the successor be scheduled once every CTA
// of this grid has issued it.
//
// launch_dependent launches so.  The rule for every kernel that it launches:
//  * pdl_wait comes before pdl_trigger and before the end, on every way through the
//    kernel.  A CTA that may run therefore knows that whatever ran before its
//    predecessor has completed: the predecessor's CTAs have all passed their own wait.
//  * Ahead of its pdl_wait a kernel writes nothing outside its CTA, and reads only what its
//    predecessor does not write: tables of the call, and what was written two launches
//    back or earlier (the sweeps after a contact pass read X, Q and the multipliers so,
//    the advance kernel Xp, Qp and, without bundles, X and Q, the later contact passes
//    and the sweeps the pair count).  A pdl_trigger moved ahead of a pdl_wait, or
//    another kernel put between, would make a race of that.
//  * What the predecessor writes is read by coherent loads after the wait: no .nc form
//    and no __ldg, which ask for memory that nothing writes while the kernel is resident.
template <typename... KArgs, typename... Args>
inline void launch_dependent(void (*kernel)(KArgs...), int grid, int block, int smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Two float4 on a 32-byte boundary in one 256-bit load (sm_100 and later): one request
// per lane for a gather of 32-byte records, instead of two.  Coherent, and not moved
// across a pdl_wait: the records (pill packs, skinning frames) are written by the
// kernel before, which a programmatic launch overlaps.
__device__ __forceinline__ void ld_record(const float4 *p, float4 &a, float4 &b)
{
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                 : "l"(p)
                 : "memory");
}

// ================================================================ rods
// Pin target in the rod's local frame.  Bone pose at substep fraction tau:
// normalised lerp of the (sign-aligned) rotations and lerp of the origins
// between the previous and target poses.  pins[2p] = (offset, bone),
// pins[2p+1] = (origin of the pinned vertex's rod, 0).
__device__ __forceinline__ V3 pin_target(const Params &P, int pin, float tau)
{
    float4 pd = P.pins[2 * pin];
    V3 o = xyz(P.pins[2 * pin + 1]);
    int b = __float2int_rn(pd.w);
    if (b < 0) return xyz(pd) - o;
    float4 q0 = P.bq0[b], q1 = P.bq1[b];
    float d = q0.x * q1.x + q0.y * q1.y + q0.z * q1.z + q0.w * q1.w;
    float sg = d < 0.f ? -1.f : 1.f;
    float t = tau, u = 1.f - t;
    float4 q = qnormalize(make_float4(u * q0.x + t * sg * q1.x, u * q0.y + t * sg * q1.y,
                                      u * q0.z + t * sg * q1.z, u * q0.w + t * sg * q1.w));
    const float *t0 = P.bt0 + 3 * b, *t1 = P.bt1 + 3 * b;
    V3 tr = {u * t0[0] + t * t1[0], u * t0[1] + t * t1[1], u * t0[2] + t * t1[2]};
    return (qrot(q, xyz(pd)) + tr) - o;
}

// Warm start from the bones (Sec. 8.2): before a frame's first substep, vertex
// v of a rod pinned at both ends to bones b0, b1 moves by linear blend skinning
// with those bones' transforms relative to their previous poses,
// T_b(p) = R1 R0^T (p - t0) + t1, with weights (1 - t, t), t the vertex's rest
// arclength fraction.  Positions only (scale, velocities and frames unchanged).
__device__ __forceinline__ float4 warm_vertex(const Params &P, int v, float4 x)
{
    const float4 wv = P.warm[v];
    if (wv.x < 0.f) return x;
    const float4 o = P.rod_origin[P.rod_of_v[v]];
    const V3 p = {x.x + o.x, x.y + o.y, x.z + o.z};
    V3 acc = {0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int b = __float2int_rn(k ? wv.y : wv.x);
        const float wk = k ? wv.z : 1.f - wv.z;
        const float *t0 = P.bt0 + 3 * b, *t1 = P.bt1 + 3 * b;
        const V3 y = qrot(P.bq1[b], qrot(qconj(P.bq0[b]), p - v3(t0[0], t0[1], t0[2]))) + v3(t1[0], t1[1], t1[2]);
        acc = acc + wk * y;
    }
    x.x = acc.x - o.x;
    x.y = acc.y - o.y;
    x.z = acc.z - o.z;
    return x;
}

// World position and radius of vertex v (x + its rod's origin, scale x rest
// radius) with the operations contact_load uses: the packed form of XW.
__device__ __forceinline__ float4 world_pack(const Params &P, int v, float4 x)
{
    const float4 o = P.rod_origin[P.rod_of_v[v]];
    return make_float4(__fadd_rn(x.x, o.x), __fadd_rn(x.y, o.y), __fadd_rn(x.z, o.z), __fmul_rn(x.w, P.RV0[v].w));
}

// The pill between world-packed vertices a and b for the early-out of the
// contact pass: box[0] = (midpoint, r), box[1] = (axis d = b - a, |d|^2), r the
// larger radius padded by 1e-3 of itself and 1e-5 of the coordinates' and the
// axis's magnitude, far above the FP32 rounding of the early-out or the search.
__device__ __forceinline__ void pill_box(float4 a, float4 b, float4 *box)
{
    const V3 d = xyz(b) - xyz(a), m = 0.5f * (xyz(a) + xyz(b));
    const float r = fmaxf(a.w, b.w), dd = dot(d, d);
    const float mag = fmaxf(fmaxf(fabsf(m.x), fabsf(m.y)), fabsf(m.z)) + fabsf(d.x) + fabsf(d.y) + fabsf(d.z);
    box[0] = make_float4(m.x, m.y, m.z, r + 1e-3f * fabsf(r) + 1e-5f * mag);
    box[1] = make_float4(d.x, d.y, d.z, dd);
}

__device__ __forceinline__ float4 to_world(const Params &P, int v, float4 x)
{
    float4 o = P.rod_origin[P.rod_of_v[v]];
    return make_float4(__fadd_rn(x.x, o.x), __fadd_rn(x.y, o.y), __fadd_rn(x.z, o.z), x.w);
}

// x_hat = x + h v + h^2 g (pinned: bone target at substep fraction tau); s_hat = s + h sdot.
__device__ __forceinline__ float4 predict_vertex(const Params &P, float4 x, float4 vel, float4 rv1, float tau)
{
    if (rv1.x < 0.f) {
        V3 t = pin_target(P, __float2int_rn(-rv1.x) - 1, tau);
        x.x = t.x;
        x.y = t.y;
        x.z = t.z;
    } else {
        const float h = P.h, hh = P.h * P.h;
        x.x += h * vel.x + hh * P.gx;
        x.y += h * vel.y + hh * P.gy;
        x.z += h * vel.z + hh * P.gz;
    }
    x.w += P.h * vel.w;
    return x;
}

__device__ __forceinline__ float4 predict_quat(const Params &P, float4 q, float4 w)
{
    rotate_by(q, P.h * xyz(w));
    return q;
}

__device__ __forceinline__ float4 omega_of(const Params &P, float4 q, float4 qp)
{
    float4 d = qmul(q, qconj(qp));
    float sg = d.w < 0.f ? -2.f : 2.f;
    return make_float4(sg * d.x * P.inv_h, sg * d.y * P.inv_h, sg * d.z * P.inv_h, 0.f);
}

__device__ __forceinline__ void check_finite(const Params &P, float4 a)
{
    if (!isfinite(a.x + a.y + a.z + a.w)) atomicOr(P.err, ERR_NONFINITE);
}

__device__ __forceinline__ float4 apply_pending(const Params &P, int v, float4 x)
{
    int c = P.cnt[v];
    if (c) {
        if (c > kFixMaxCount) atomicOr(P.err, ERR_CONTACTS);  // the field sums may have wrapped
        const float inv = 1.f / (float)c;
        unsigned long long *a = P.acc + 2 * (size_t)v;
        float dx, dy, dz, dr;
        fix_unpack(a[0], P.fix_inv, dx, dy);
        fix_unpack(a[1], P.fix_inv, dz, dr);
        x.x += dx * inv;
        x.y += dy * inv;
        x.z += dz * inv;
        const float rb = P.RV0[v].w;  // the radius change back to a scale change
        if (rb > 0.f) x.w += (dr / rb) * inv;
        a[0] = a[1] = 0ull;
        P.cnt[v] = 0;
    }
    return x;
}

// ---------------------------------------------------------------- element phases
// Prediction of vertex v at substep fraction tau (Sec. 6): keeps the substep's
// start in Xp, writes the predicted world position for the broadphase when
// `world`, clears the half-plane multipliers and, when `plain_lam`, the
// per-constraint multipliers of the launch-per-colour kernels.
__device__ __forceinline__ void predict_vertex_at(const Params &P, int v, float tau, bool world, bool plain_lam)
{
    float4 x = P.X[v];
    P.Xp[v] = x;
    x = predict_vertex(P, x, P.V[v], P.RV1[v], tau);
    P.X[v] = x;
    if (world) P.Xpred[v] = to_world(P, v, x);
    if (plain_lam) {
        P.lamB[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        P.lamB2[v] = 0.f;
        P.lamL[v] = 0.f;
    }
    for (int k = 0; k < P.n_planes; ++k) P.lam_plane[(size_t)v * P.n_planes + k] = 0.f;
}

__device__ __forceinline__ void predict_segment_at(const Params &P, int g, bool plain_lam)
{
    float4 q = P.Q[g];
    P.Qp[g] = q;
    P.Q[g] = predict_quat(P, q, P.W[g]);
    if (plain_lam) {
        P.lamS[g] = make_float4(0.f, 0.f, 0.f, 0.f);
        P.lamS2[g] = make_float2(0.f, 0.f);
        if (P.vvec) P.lamV2[g] = make_float2(0.f, 0.f);
    }
}

// The start of a substep for vertex v (segment g) without its first sweep: with
// `finish_prev`, the previous substep's pending contact corrections and
// velocity update; then the prediction (Sec. 6) at bone fraction tau, the
// substep's start state in Xp, the predicted world position for the
// broadphase when `world`, and cleared half-plane multipliers (as the first
// sweep kernel does before its sweep).  advance_*_load reads what the last
// contact pass does not change (`state`: the positions and frames too, which
// shape matching and the warm start do change), and works out a pinned vertex's
// target; advance_*_at does the rest.
struct AdvanceVertex {
    float4 x, xp, vel, rv1, o;
    V3 pin;
};
__device__ __forceinline__ void advance_vertex_load(const Params &P, int v, bool finish_prev, bool state, float tau,
                                                    bool world, AdvanceVertex &A)
{
    A.rv1 = P.RV1[v];
    if (state) A.x = P.X[v];
    if (finish_prev)
        A.xp = P.Xp[v];
    else
        A.vel = P.V[v];
    if (world) A.o = P.rod_origin[P.rod_of_v[v]];
    if (A.rv1.x < 0.f) A.pin = pin_target(P, __float2int_rn(-A.rv1.x) - 1, tau);
}

__device__ __forceinline__ void advance_vertex_at(const Params &P, int v, bool finish_prev, bool state, bool world,
                                                  AdvanceVertex &A)
{
    float4 x = state ? A.x : P.X[v];
    float4 vel = A.vel;
    if (finish_prev) {
        x = apply_pending(P, v, x);
        const float4 xp = A.xp;
        vel = make_float4((x.x - xp.x) * P.inv_h, (x.y - xp.y) * P.inv_h, (x.z - xp.z) * P.inv_h,
                          (x.w - xp.w) * P.inv_h);
        check_finite(P, x);
        P.V[v] = vel;
    }
    P.Xp[v] = x;
    if (A.rv1.x < 0.f)
        x = make_float4(A.pin.x, A.pin.y, A.pin.z, x.w + P.h * vel.w);
    else
        x = predict_vertex(P, x, vel, A.rv1, 0.f);
    if (world) P.Xpred[v] = make_float4(__fadd_rn(x.x, A.o.x), __fadd_rn(x.y, A.o.y), __fadd_rn(x.z, A.o.z), x.w);
    for (int k = 0; k < P.n_planes; ++k) P.lam_plane[(size_t)v * P.n_planes + k] = 0.f;
    P.X[v] = x;
}

struct AdvanceSegment {
    float4 q, qp, w;
};
__device__ __forceinline__ void advance_segment_load(const Params &P, int g, bool finish_prev, bool state,
                                                     AdvanceSegment &A)
{
    if (state) A.q = P.Q[g];
    if (finish_prev)
        A.qp = P.Qp[g];
    else
        A.w = P.W[g];
}

__device__ __forceinline__ void advance_segment_at(const Params &P, int g, bool finish_prev, bool state,
                                                   const AdvanceSegment &A)
{
    const float4 q = state ? A.q : P.Q[g];
    float4 w = A.w;
    if (finish_prev) {
        check_finite(P, q);
        w = omega_of(P, q, A.qp);
        P.W[g] = w;
    }
    P.Qp[g] = q;
    P.Q[g] = predict_quat(P, q, w);
}

// Velocity update of vertex v (after the pending contact corrections when `apply`).
__device__ __forceinline__ void finish_vertex_at(const Params &P, int v, bool apply)
{
    float4 x = P.X[v];
    if (apply) x = apply_pending(P, v, x);
    const float4 xp = P.Xp[v];
    const float4 vel = make_float4((x.x - xp.x) * P.inv_h, (x.y - xp.y) * P.inv_h, (x.z - xp.z) * P.inv_h,
                                   (x.w - xp.w) * P.inv_h);
    check_finite(P, x);
    P.X[v] = x;
    P.V[v] = vel;
}

__device__ __forceinline__ void finish_segment_at(const Params &P, int g)
{
    const float4 q = P.Q[g];
    check_finite(P, q);
    P.W[g] = omega_of(P, q, P.Qp[g]);
}

// A rod work item's per-element state in shared memory, de-interleaved: the
// elements with even item-local index first, then the odd ones.  A colour's
// threads touch every second element of their rods, so each colour reads and
// writes consecutive float4s (no shared-memory bank conflicts).
struct SmemRod {
    float4 *p;
    int half;  // elements with even index: (n + 1) / 2
    __device__ __forceinline__ float4 &operator[](int i) const { return p[(i & 1) ? half + (i >> 1) : (i >> 1)]; }
};
__device__ __forceinline__ SmemRod smem_rod(float4 *p, int n) { return SmemRod{p, (n + 1) >> 1}; }

// Multipliers of one slot kept across launches (contact path): 24 floats.
struct SlotLam {
    float4 s0, s1, b1, b2;
    float2 x0, x1;
    float v1, v2;
    float l1, l2;  // surface bending at vertices 2p+1, 2p+2
};

__device__ __forceinline__ void lam_load(const Params &P, int slot, SlotLam &L)
{
    const float *b = P.slot_lam + slot;
    const int st = P.slot_stride;
    float t[kSlotLam];
#pragma unroll
    for (int k = 0; k < kSlotLam - 2; ++k) t[k] = b[k * st];
    t[22] = t[23] = 0.f;
    if (P.surface) {
        t[22] = b[22 * st];
        t[23] = b[23 * st];
    }
    L.s0 = make_float4(t[0], t[1], t[2], t[3]);
    L.s1 = make_float4(t[4], t[5], t[6], t[7]);
    L.b1 = make_float4(t[8], t[9], t[10], t[11]);
    L.b2 = make_float4(t[12], t[13], t[14], t[15]);
    L.x0 = make_float2(t[16], t[17]);
    L.x1 = make_float2(t[18], t[19]);
    L.v1 = t[20];
    L.v2 = t[21];
    L.l1 = t[22];
    L.l2 = t[23];
}

__device__ __forceinline__ void lam_store(const Params &P, int slot, const SlotLam &L)
{
    float *b = P.slot_lam + slot;
    const int st = P.slot_stride;
    const float t[kSlotLam] = {L.s0.x, L.s0.y, L.s0.z, L.s0.w, L.s1.x, L.s1.y, L.s1.z, L.s1.w,
                               L.b1.x, L.b1.y, L.b1.z, L.b1.w, L.b2.x, L.b2.y, L.b2.z, L.b2.w,
                               L.x0.x, L.x0.y, L.x1.x, L.x1.y, L.v1, L.v2, L.l1, L.l2};
#pragma unroll
    for (int k = 0; k < kSlotLam - 2; ++k) b[k * st] = t[k];
    if (P.surface) {
        b[22 * st] = t[22];
        b[23 * st] = t[23];
    }
}


// The constraints one thread owns in the shared-memory rod kernels: segments
// 2p, 2p+1 and interior vertices 2p+1, 2p+2 of one rod (slot p), with their
// rest data held in registers.
struct SlotRest {
    bool active, has0, has1, hasv2;
    int lv, ls;  // local first vertex / segment of the slot inside the item
    int gv;      // global index of vertex 2p
    int p2;      // 2p: rod-local index of vertex 2p
    int n;       // vertices of the slot's rod
    float4 rs00, rs01, rv01, rv02;
    float2 rs10, rs11;
    float w0, w1, w2, ws0, ws1, ws2, ws3, aB1, aV1, aB2, aV2, l2, im2;
};

__device__ __forceinline__ void load_slot(const Params &P, int4 item, int2 sd, SlotRest &R)
{
    R.active = sd.y >= 0;
    const int vb = sd.x & 0xffff, N = R.active ? (sd.x >> 16) : 0;
    const int sb = sd.y & 0xffff, p = R.active ? (sd.y >> 16) : 0;
    R.lv = vb + 2 * p;
    R.ls = sb + 2 * p;
    const int gv = item.x + R.lv, gs = item.z + R.ls;
    R.gv = gv;
    R.p2 = 2 * p;
    R.n = N;
    R.has0 = R.active;
    R.has1 = R.active && (2 * p + 1 <= N - 2);   // segment 2p+1 and vertex 2p+1
    R.hasv2 = R.active && (2 * p + 2 <= N - 2);  // vertex 2p+2
    R.rs00 = make_float4(1.f, 0.f, 0.f, 0.f);
    R.rs01 = R.rs00;
    R.rv01 = make_float4(0.f, 0.f, 0.f, 0.f);
    R.rv02 = R.rv01;
    R.rs10 = make_float2(0.f, 0.f);
    R.rs11 = R.rs10;
    R.w0 = R.w1 = R.w2 = R.ws0 = R.ws1 = R.ws2 = R.ws3 = 0.f;
    R.aB1 = R.aV1 = R.aB2 = R.aV2 = 0.f;
    R.l2 = 1.f;
    R.im2 = 0.f;
    if (R.has0) {
        R.rs00 = P.RS0[gs];
        R.rs10 = P.RS1[gs];
        float4 r0 = P.RV1[gv], r1 = P.RV1[gv + 1];
        R.w0 = inv_mass(r0);
        R.ws0 = r0.y;
        R.w1 = inv_mass(r1);
        R.ws1 = r1.y;
        R.aB1 = r1.z;
        R.aV1 = r1.w;
    }
    if (R.has1) {
        R.rs01 = P.RS0[gs + 1];
        R.rs11 = P.RS1[gs + 1];
        float4 r2 = P.RV1[gv + 2];
        R.w2 = inv_mass(r2);
        R.ws2 = r2.y;
        R.aB2 = r2.z;
        R.aV2 = r2.w;
        R.rv01 = P.RV0[gv + 1];
    }
    if (R.hasv2) {
        float4 r = P.RS0[gs + 2];
        R.l2 = r.x;
        R.im2 = r.y;
        R.rv02 = P.RV0[gv + 2];
        if (P.surface) R.ws3 = P.RV1[gv + 3].y;
    }
}

__device__ __forceinline__ void zero_lam(SlotLam &L)
{
    L.s0 = L.s1 = L.b1 = L.b2 = make_float4(0.f, 0.f, 0.f, 0.f);
    L.x0 = L.x1 = make_float2(0.f, 0.f);
    L.v1 = L.v2 = 0.f;
    L.l1 = L.l2 = 0.f;
}

// One sweep of the four colours over the item staged in shared memory, then,
// with surface bending (RV2 non-null), three colours of interior vertices
// i mod 3 (each couples scales i-1, i, i+1).  Every thread of the CTA must call
// it (it synchronises the CTA between colours).
__device__ __forceinline__ void sweep(SmemRod sX, SmemRod sQ, const SlotRest &R, SlotLam &L, float inv_h2,
                                      bool vol, const float4 *__restrict__ RV2 = nullptr)
{
    const int lv = R.lv;
    // the slot's elements: of one parity they lie side by side (SmemRod)
    float4 *const x0 = &sX[lv], *const x1 = &sX[lv + 1], *const q0 = &sQ[R.ls], *const q1 = &sQ[R.ls + 1];
    // colour 0: even segments
    if (R.has0) {
        float4 xa = x0[0], xb = x1[0], q = q0[0];
        project_segment(xa, xb, q, R.w0, R.w1, R.ws0, R.ws1, R.rs00, R.rs10, L.s0, L.x0, inv_h2, vol);
        x0[0] = xa;
        x1[0] = xb;
        q0[0] = q;
    }
    __syncthreads();
    // colour 1: odd segments
    if (R.has1) {
        float4 xa = x1[0], xb = x0[1], q = q1[0];
        project_segment(xa, xb, q, R.w1, R.w2, R.ws1, R.ws2, R.rs01, R.rs11, L.s1, L.x1, inv_h2, vol);
        x1[0] = xa;
        x0[1] = xb;
        q1[0] = q;
    }
    __syncthreads();
    // colour 2: even interior vertices (2p+2), segments 2p+1 and 2p+2
    if (R.hasv2) {
        float4 qa = q1[0], qb = q0[1];
        float s = x0[1].w;
        project_vertex(qa, qb, s, x1[0].w, x1[1].w, R.rs01.x, R.l2, R.rs01.y, R.im2, R.ws2, R.rv02, R.aB2, R.aV2,
                       L.b2, L.v2, inv_h2, vol);
        q1[0] = qa;
        q0[1] = qb;
        x0[1].w = s;
    }
    __syncthreads();
    // colour 3: odd interior vertices (2p+1), segments 2p and 2p+1
    if (R.has1) {
        float4 qa = q0[0], qb = q1[0];
        float s = x1[0].w;
        project_vertex(qa, qb, s, x0[0].w, x0[1].w, R.rs00.x, R.rs01.x, R.rs00.y, R.rs01.y, R.ws1, R.rv01, R.aB1,
                       R.aV1, L.b1, L.v1, inv_h2, vol);
        q0[0] = qa;
        q1[0] = qb;
        x1[0].w = s;
    }
    __syncthreads();
    if (RV2) {
        // the slot's two vertices fall on different colours: a colour takes one of them
        // (none: lap = 0), by selection, so that a warp runs the constraint once per
        // colour; what does not depend on the scales is worked out before.
        // 1,021 rods, a frame 184 -> 173 us.
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 ra = R.has1 ? __ldg(RV2 + R.gv + 1) : z, rb = R.hasv2 ? __ldg(RV2 + R.gv + 2) : z;
        const LapRest A = lap_rest(ra, R.ws0, R.ws1, R.ws2, inv_h2), B = lap_rest(rb, R.ws1, R.ws2, R.ws3, inv_h2);
        const int c1 = R.has1 ? (R.p2 + 1) % 3 : 3, c2 = R.hasv2 ? (R.p2 + 2) % 3 : 3;
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
            const int lap = c == c1 ? 1 : c == c2 ? 2 : 0;
            if (lap) {
                const bool one = lap == 1;
                const int v = lv + lap;
                LapRest T;
                T.jp = one ? A.jp : B.jp;
                T.jn = one ? A.jn : B.jn;
                T.at = one ? A.at : B.at;
                T.inv = one ? A.inv : B.inv;
                const float wp = one ? R.ws0 : R.ws1, w = one ? R.ws1 : R.ws2, wn = one ? R.ws2 : R.ws3;
                float sp = sX[v - 1].w, s = sX[v].w, sn = sX[v + 1].w, lam = one ? L.l1 : L.l2;
                project_laplacian(sp, s, sn, wp, w, wn, T, lam);
                sX[v - 1].w = sp;
                sX[v].w = s;
                sX[v + 1].w = sn;
                if (one)
                    L.l1 = lam;
                else
                    L.l2 = lam;
            }
            __syncthreads();
        }
    }
}

// One Jacobi-with-averaging iteration over the item staged in shared memory
// (Sec. 7 engine): every constraint is evaluated on the iteration's starting
// state with its own multiplier; the increments go to per-constraint records
// in shared memory (jS: 3 float4 per segment, jV: 2 per vertex, jL: 1 per
// vertex with surface bending); then each thread moves the degrees of freedom
// it owns (vertices 2p, 2p+1 and the rod's last one, segments 2p, 2p+1) by the
// sum of the records acting on them divided by their number.  Every thread
// of the CTA must call it.
__device__ __forceinline__ void sweep_jacobi(SmemRod sX, SmemRod sQ, const SlotRest &R, SlotLam &L, float inv_h2,
                                             bool vol, const float4 *__restrict__ RV2, float4 *jS, float4 *jV,
                                             float4 *jL)
{
    const int lv = R.lv, ls = R.ls;
    // ---- every constraint on the starting state
    if (R.has0) {
        SegDelta d;
        jacobi_segment(sX[lv], sX[lv + 1], sQ[ls], R.w0, R.w1, R.ws0, R.ws1, R.rs00, R.rs10, L.s0, L.x0, inv_h2, vol,
                       d);
        jS[3 * ls] = make_float4(d.dxa.x, d.dxa.y, d.dxa.z, d.dsa);
        jS[3 * ls + 1] = make_float4(d.dxb.x, d.dxb.y, d.dxb.z, d.dsb);
        jS[3 * ls + 2] = make_float4(d.dth.x, d.dth.y, d.dth.z, 0.f);
    }
    if (R.has1) {
        SegDelta d;
        jacobi_segment(sX[lv + 1], sX[lv + 2], sQ[ls + 1], R.w1, R.w2, R.ws1, R.ws2, R.rs01, R.rs11, L.s1, L.x1,
                       inv_h2, vol, d);
        jS[3 * (ls + 1)] = make_float4(d.dxa.x, d.dxa.y, d.dxa.z, d.dsa);
        jS[3 * (ls + 1) + 1] = make_float4(d.dxb.x, d.dxb.y, d.dxb.z, d.dsb);
        jS[3 * (ls + 1) + 2] = make_float4(d.dth.x, d.dth.y, d.dth.z, 0.f);
        // vertex 2p+1 between segments 2p and 2p+1
        VtxDelta e;
        jacobi_vertex(sQ[ls], sQ[ls + 1], sX[lv + 1].w, sX[lv].w, sX[lv + 2].w, R.rs00.x, R.rs01.x, R.rs00.y,
                      R.rs01.y, R.ws1, R.rv01, R.aB1, R.aV1, L.b1, L.v1, inv_h2, vol, e);
        jV[2 * (lv + 1)] = make_float4(e.dtha.x, e.dtha.y, e.dtha.z, e.ds);
        jV[2 * (lv + 1) + 1] = make_float4(e.dthb.x, e.dthb.y, e.dthb.z, 0.f);
        if (RV2) {
            float dsp, ds, dsn;
            laplacian_increments(sX[lv].w, sX[lv + 1].w, sX[lv + 2].w, R.ws0, R.ws1, R.ws2, __ldg(RV2 + R.gv + 1),
                                 L.l1, inv_h2, dsp, ds, dsn);
            jL[lv + 1] = make_float4(dsp, ds, dsn, 0.f);
        }
    }
    if (R.hasv2) {  // vertex 2p+2 between segments 2p+1 and 2p+2
        VtxDelta e;
        jacobi_vertex(sQ[ls + 1], sQ[ls + 2], sX[lv + 2].w, sX[lv + 1].w, sX[lv + 3].w, R.rs01.x, R.l2, R.rs01.y,
                      R.im2, R.ws2, R.rv02, R.aB2, R.aV2, L.b2, L.v2, inv_h2, vol, e);
        jV[2 * (lv + 2)] = make_float4(e.dtha.x, e.dtha.y, e.dtha.z, e.ds);
        jV[2 * (lv + 2) + 1] = make_float4(e.dthb.x, e.dthb.y, e.dthb.z, 0.f);
        if (RV2) {
            float dsp, ds, dsn;
            laplacian_increments(sX[lv + 1].w, sX[lv + 2].w, sX[lv + 3].w, R.ws1, R.ws2, R.ws3,
                                 __ldg(RV2 + R.gv + 2), L.l2, inv_h2, dsp, ds, dsn);
            jL[lv + 2] = make_float4(dsp, ds, dsn, 0.f);
        }
    }
    __syncthreads();
    // ---- each owner averages the records acting on its degrees of freedom
    if (R.active) {
        const int N = R.n, vb = lv - R.p2, sb = ls - R.p2;  // the rod's first vertex / segment in the item
        const float nS = vol ? 2.f : 1.f;   // S, V on positions and on the frame
        const float nSs = vol ? 3.f : 2.f;  // V, X, G on scales
        const float nB = vol ? 2.f : 1.f;   // B, Vb on the vertex scale and both frames
        const int last = (R.p2 + 2 == N - 1) ? 3 : 2;
        for (int k = 0; k < last; ++k) {
            const int i = R.p2 + k;  // rod-local vertex
            V3 dx = v3(0.f, 0.f, 0.f);
            float ds = 0.f, cx = 0.f, cs = 0.f;
            if (i >= 1) {
                const float4 b = jS[3 * (sb + i - 1) + 1];
                dx = dx + xyz(b);
                ds += b.w;
                cx += nS;
                cs += nSs;
            }
            if (i <= N - 2) {
                const float4 a = jS[3 * (sb + i)];
                dx = dx + xyz(a);
                ds += a.w;
                cx += nS;
                cs += nSs;
            }
            if (i >= 1 && i <= N - 2) {
                ds += jV[2 * (vb + i)].w;
                cs += nB;
            }
            if (RV2) {
                if (i - 1 >= 1) { ds += jL[vb + i - 1].z; cs += 1.f; }
                if (i >= 1 && i <= N - 2) { ds += jL[vb + i].y; cs += 1.f; }
                if (i + 1 <= N - 2) { ds += jL[vb + i + 1].x; cs += 1.f; }
            }
            float4 x = sX[vb + i];
            add_to(x, (1.f / cx) * dx);
            x.w += ds / cs;
            sX[vb + i] = x;
        }
        for (int k = 0; k < 2; ++k) {
            const int j = R.p2 + k;  // rod-local segment
            if (j > N - 2) break;
            const float4 t = jS[3 * (sb + j) + 2];
            V3 dth = xyz(t);
            float cq = nS;
            if (j >= 1) {
                dth = dth + xyz(jV[2 * (vb + j) + 1]);
                cq += nB;
            }
            if (j + 1 <= N - 2) {
                dth = dth + xyz(jV[2 * (vb + j + 1)]);
                cq += nB;
            }
            float4 q = sQ[sb + j];
            rotate_by(q, (1.f / cq) * dth);
            sQ[sb + j] = q;
        }
    }
    __syncthreads();
}

// The iteration of either ordering.  rec: the shared-memory records of
// sweep_jacobi (3 float4 per segment, 3 per vertex), unused by the colours.
__device__ __forceinline__ void sweep_any(const Params &P, SmemRod sX, SmemRod sQ, const SlotRest &R, SlotLam &L,
                                          float4 *rec, int4 item)
{
    const bool vol = P.volume != 0;
    const float4 *RV2 = P.surface ? P.RV2 : nullptr;
    if (P.jacobi) {
        float4 *jS = rec, *jV = rec + 3 * item.w, *jL = jV + 2 * item.y;
        sweep_jacobi(sX, sQ, R, L, P.inv_h2, vol, RV2, jS, jV, jL);
    } else {
        sweep(sX, sQ, R, L, P.inv_h2, vol, RV2);
    }
}

// One sweep of one work item between contact passes, in two parts.  rod_stage: a
// CTA stages the item's float4 state in shared memory with coalesced loads and
// each thread's rest data and multipliers in registers.  rod_run adds the pending
// contact corrections when `apply`, runs a sweep and writes the state back.  Item
// b's slot descriptors and multipliers are entries b * blockDim.x + threadIdx.x.
// Every thread of the CTA calls both.  A contact pass changes nothing that
// rod_stage reads, so the sweep after it can stage while the pass still runs.
struct RodStage {
    int4 item;
    int slot;
    SlotRest R;
    SlotLam L;
};

__device__ __forceinline__ void rod_stage_rest(const Params &P, int b, bool first, RodStage &S)
{
    S.item = P.items[b];
    S.slot = b * blockDim.x + threadIdx.x;
    load_slot(P, S.item, P.slots[S.slot], S.R);
    if (first)
        zero_lam(S.L);
    else
        lam_load(P, S.slot, S.L);
}

__device__ __forceinline__ void rod_stage_state(const Params &P, const RodStage &S, float4 *smem)
{
    const int4 item = S.item;
    const SmemRod sX = smem_rod(smem, item.y);
    const SmemRod sQ = smem_rod(smem + item.y, item.w);
    for (int i = threadIdx.x; i < item.y; i += blockDim.x) sX[i] = P.X[item.x + i];
    for (int j = threadIdx.x; j < item.w; j += blockDim.x) sQ[j] = P.Q[item.z + j];
}

__device__ __forceinline__ void rod_run(const Params &P, RodStage &S, bool apply, float4 *smem)
{
    const int4 item = S.item;
    const SmemRod sX = smem_rod(smem, item.y);
    const SmemRod sQ = smem_rod(smem + item.y, item.w);
    if (apply)  // to the elements this thread staged
        for (int i = threadIdx.x; i < item.y; i += blockDim.x) sX[i] = apply_pending(P, item.x + i, sX[i]);
    __syncthreads();
    sweep_any(P, sX, sQ, S.R, S.L, smem + 2 * (item.y + item.w), item);  // Jacobi records behind the state
    if (S.R.active) lam_store(P, S.slot, S.L);

    for (int i = threadIdx.x; i < item.y; i += blockDim.x) {
        const int v = item.x + i;
        const float4 x = sX[i];
        P.X[v] = x;
        if (P.XW) {
            const float4 xw = world_pack(P, v, x);
            P.XW[v] = xw;
            // the pill from v on (after a rod's last vertex: not a pill, and not read)
            if (i + 1 < item.y) pill_box(xw, world_pack(P, v + 1, sX[i + 1]), P.PB + 2 * (size_t)v);
        }
    }
    for (int j = threadIdx.x; j < item.w; j += blockDim.x) P.Q[item.z + j] = sQ[j];
}

// A whole frame of one work item of a scene without contacts: nothing couples
// its rods to others, so the CTA keeps their state in shared memory, and their
// rest data in registers, from the first substep to the last.  The velocity of a
// substep is that of its predecessor, from the positions still in shared memory.
// Against a launch per substep, with the state staged and the rest data loaded
// each time: 16 rods of 32 vertices, two frames of 10 substeps 268 -> 226 us; 4,096
// rods of 4 to 256 vertices, a frame of 20 substeps 1,486 -> 1,373 us.
__device__ __forceinline__ void rod_frame_item(const Params &P, int b, int substeps, int n_iter, float4 *smem)
{
    const int4 item = P.items[b];
    const SmemRod sX = smem_rod(smem, item.y);
    const SmemRod sQ = smem_rod(smem + item.y, item.w);
    const SmemRod sXp = smem_rod(smem + item.y + item.w, item.y);
    const SmemRod sQp = smem_rod(smem + 2 * item.y + item.w, item.w);
    float4 *rec = smem + 2 * (item.y + item.w);  // Jacobi records behind the state
    for (int i = threadIdx.x; i < item.y; i += blockDim.x) sX[i] = P.X[item.x + i];
    for (int j = threadIdx.x; j < item.w; j += blockDim.x) sQ[j] = P.Q[item.z + j];
    SlotRest R;
    load_slot(P, item, P.slots[b * blockDim.x + threadIdx.x], R);
    // the thread that loaded an element also predicts it and writes it back
    auto vel_of = [&](float4 x, float4 xp) {
        return make_float4((x.x - xp.x) * P.inv_h, (x.y - xp.y) * P.inv_h, (x.z - xp.z) * P.inv_h,
                           (x.w - xp.w) * P.inv_h);
    };
#pragma unroll 1
    for (int k = 0; k < substeps; ++k) {
        const float tau = (float)((double)(k + 1) / substeps);
        for (int i = threadIdx.x; i < item.y; i += blockDim.x) {
            const int v = item.x + i;
            const float4 x = sX[i];
            float4 vel;
            if (k) {
                check_finite(P, x);
                vel = vel_of(x, sXp[i]);
            } else {
                vel = P.V[v];
            }
            sXp[i] = x;
            sX[i] = predict_vertex(P, x, vel, P.RV1[v], tau);
        }
        for (int j = threadIdx.x; j < item.w; j += blockDim.x) {
            const float4 q = sQ[j];
            float4 w;
            if (k) {
                check_finite(P, q);
                w = omega_of(P, q, sQp[j]);
            } else {
                w = P.W[item.z + j];
            }
            sQp[j] = q;
            sQ[j] = predict_quat(P, q, w);
        }
        SlotLam L;
        zero_lam(L);
        __syncthreads();
#pragma unroll 1
        for (int it = 0; it < n_iter; ++it) sweep_any(P, sX, sQ, R, L, rec, item);
    }
    for (int i = threadIdx.x; i < item.y; i += blockDim.x) {
        const float4 x = sX[i];
        check_finite(P, x);
        P.V[item.x + i] = vel_of(x, sXp[i]);
        P.X[item.x + i] = x;
    }
    for (int j = threadIdx.x; j < item.w; j += blockDim.x) {
        const float4 q = sQ[j];
        check_finite(P, q);
        P.W[item.z + j] = omega_of(P, q, sQp[j]);
        P.Q[item.z + j] = q;
    }
}

// First sweep of a substep on the contact path, for one work item: the
// previous substep's velocity update (after its last contact pass) when
// finish_prev, the prediction (Sec. 6) -- the start state kept in Xp / Qp,
// the predicted world positions in Xpred when `world`, the half-plane
// multipliers cleared -- then one colour sweep with fresh multipliers.
// The same per-element arithmetic as finish_*_at, predict_*_at and rod_run.
__device__ __forceinline__ void rod_item_first(const Params &P, int b, bool finish_prev, float tau, bool world,
                                               float4 *smem)
{
    const int4 item = P.items[b];
    const SmemRod sX = smem_rod(smem, item.y);
    const SmemRod sQ = smem_rod(smem + item.y, item.w);
    for (int i = threadIdx.x; i < item.y; i += blockDim.x) {
        const int v = item.x + i;
        float4 x = P.X[v], vel;
        if (finish_prev) {
            x = apply_pending(P, v, x);
            const float4 xp = P.Xp[v];
            vel = make_float4((x.x - xp.x) * P.inv_h, (x.y - xp.y) * P.inv_h, (x.z - xp.z) * P.inv_h,
                              (x.w - xp.w) * P.inv_h);
            check_finite(P, x);
            P.V[v] = vel;
        } else {
            vel = P.V[v];
        }
        P.Xp[v] = x;
        x = predict_vertex(P, x, vel, P.RV1[v], tau);
        if (world) P.Xpred[v] = to_world(P, v, x);
        for (int k = 0; k < P.n_planes; ++k) P.lam_plane[(size_t)v * P.n_planes + k] = 0.f;
        sX[i] = x;
    }
    for (int j = threadIdx.x; j < item.w; j += blockDim.x) {
        const int g = item.z + j;
        const float4 q = P.Q[g];
        float4 w;
        if (finish_prev) {
            check_finite(P, q);
            w = omega_of(P, q, P.Qp[g]);
            P.W[g] = w;
        } else {
            w = P.W[g];
        }
        P.Qp[g] = q;
        sQ[j] = predict_quat(P, q, w);
    }
    const int slot = b * blockDim.x + threadIdx.x;
    SlotRest R;
    load_slot(P, item, P.slots[slot], R);
    SlotLam L;
    zero_lam(L);
    __syncthreads();
    sweep_any(P, sX, sQ, R, L, smem + 2 * (item.y + item.w), item);
    if (R.active) lam_store(P, slot, L);
    for (int i = threadIdx.x; i < item.y; i += blockDim.x) P.X[item.x + i] = sX[i];
    for (int j = threadIdx.x; j < item.w; j += blockDim.x) P.Q[item.z + j] = sQ[j];
}

// ================================================================ broadphase helpers
// ---------------------------------------------------------------- ordered float encoding
__device__ __forceinline__ unsigned int ord_enc(float f)
{
    unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord_dec(unsigned int u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Grid from the bounds: cell = 2 r_cut (1 + 2^-8) with r_cut the largest
// bounding radius (or, in the multi-kernel broadphase, the cut radius below
// which all but a bounded number of pills lie); grown until the dense grid
// fits the table and spans at most 4096 cells per axis.  Non-finite bounds
// (a diverged state) give an empty grid and raise the non-finite flag.
//
// `split`: cells may be cut along x, into four or two where the table has room
// (inv_x): a pill searches the part of a row of cells that its reach covers
// (emit_pills), so thinner cells leave out more of it.  Settled strands: 211
// candidates a pill, 159 with cells cut in four.
__device__ __forceinline__ Grid make_grid_from(const unsigned int *bounds, int table, bool &ok, float r_cut = -1.f,
                                               int b_cut = kRadBins - 1, bool split = false)
{
    Grid G;
    float lo[3], hi[3];
    ok = true;
    for (int c = 0; c < 3; ++c) {
        lo[c] = -ord_dec(bounds[c]);
        hi[c] = ord_dec(bounds[3 + c]);
        ok = ok && isfinite(lo[c]) && isfinite(hi[c]) && hi[c] >= lo[c];
    }
    if (!(r_cut >= 0.f)) r_cut = ord_dec(bounds[6]);
    G.r_cut = r_cut;
    G.b_cut = b_cut;
    float cell = 2.f * r_cut * 1.00390625f;
    ok = ok && isfinite(cell);
    if (!ok) {
        for (int c = 0; c < 3; ++c) {
            G.lo[c] = 0.f;
            G.dim[c] = 1;
        }
        G.inv_cell = G.inv_x = 0.f;
        G.pad = 1;
        return G;
    }
    float ext = fmaxf(fmaxf(hi[0] - lo[0], hi[1] - lo[1]), hi[2] - lo[2]);
    cell = fmaxf(cell, ext * (1.f / 4096.f));
    cell = fmaxf(cell, 1e-30f);
    int dim[3];
    for (int k = 0; k < 200; ++k) {
        float inv = 1.f / cell;
        long long tot = 1;
        for (int c = 0; c < 3; ++c) {
            dim[c] = (int)floorf((hi[c] - lo[c]) * inv) + 1;
            if (dim[c] < 1) dim[c] = 1;
            tot *= dim[c];
        }
        G.inv_cell = G.inv_x = inv;
        if (tot <= (long long)table) break;
        cell *= 1.26f;
    }
    for (int f = 4; split && f > 1; f >>= 1) {
        const float inv = f * G.inv_cell;
        const int n = (int)floorf((hi[0] - lo[0]) * inv) + 1;
        if (n > 0 && (long long)n * dim[1] * dim[2] <= (long long)table) {
            G.inv_x = inv;
            dim[0] = n;
            break;
        }
    }
    for (int c = 0; c < 3; ++c) {
        G.lo[c] = lo[c];
        G.dim[c] = dim[c];
    }
    G.pad = 0;
    return G;
}

__device__ __forceinline__ Grid make_grid(const Params &P, bool &ok) { return make_grid_from(P.bounds, P.table, ok); }

// Cells the grid spans (at most n, the table size); cells beyond stay empty.
__device__ __forceinline__ int grid_cells(const Grid *g, int n)
{
    const long long t = (long long)g->dim[0] * g->dim[1] * g->dim[2];
    return t < n ? (int)t : n;
}

__device__ __forceinline__ int cell_coord(float x, float lo, float inv_cell, int dim)
{
    int i = (int)floorf((x - lo) * inv_cell);
    return min(max(i, 0), dim - 1);
}

// Cells along an axis that hold every centre within `reach` of x.  Measured, as the
// centres' own cells are, by the rounded offset d = x - lo into the grid, and enlarged
// for the rounding: by 2^-8 of the reach for that of the radii and of the overlap test,
// and by 2^-21 of the offset, eight times the largest rounding of d and of the partner's
// offset.  (The second counts where the grid spans more than 2^15 times the reach: of
// pairs of 5 mm pills near tangency at cell borders, 1 per cent lay outside without it
// in a grid of 10 km, 24 in one of 100 km.)
__device__ __forceinline__ void cell_range(float x, float reach, float lo, float inv_cell, int dim, int &c0, int &c1)
{
    const float d = __fsub_rn(x, lo);
    const float r = __fadd_rn(__fmul_rn(reach, 1.00390625f), __fmul_rn(fabsf(d), 0x1p-21f));
    c0 = min(max((int)floorf(__fmul_rn(__fsub_rn(d, r), inv_cell)), 0), dim - 1);
    c1 = min(max((int)floorf(__fmul_rn(__fadd_rn(d, r), inv_cell)), 0), dim - 1);
}

__device__ __forceinline__ int warp_incl_scan(int v)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) >= o) v += t;
    }
    return v;
}

// exclusive scan of one value per thread across the block; returns the block total in *total
__device__ __forceinline__ int block_excl_scan(int v, int *warp_sums, int *total)
{
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = warp_incl_scan(v);
    if (lane == 31) warp_sums[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int nw = blockDim.x >> 5;
        int w = lane < nw ? warp_sums[lane] : 0;
        int wi = warp_incl_scan(w);
        if (lane < nw) warp_sums[lane] = wi - w;
        if (lane == nw - 1) warp_sums[32] = wi;
    }
    __syncthreads();
    int r = warp_sums[wid] + inc - v;
    *total = warp_sums[32];
    __syncthreads();
    return r;
}


// Bounding sphere of pill g from the predicted world state (see pill_sphere).
__device__ __forceinline__ float4 bp_sphere(const Params &P, int g)
{
    const int a = P.seg_v0[g];
    const float ra = P.bp_rbar[(size_t)a * P.bp_rbar_stride], rb = P.bp_rbar[(size_t)(a + 1) * P.bp_rbar_stride];
    return pill_sphere(P.Xpred[a], ra, P.Xpred[a + 1], rb);
}

__device__ __forceinline__ int bp_cell(const Grid &G, float4 sp)
{
    const int ix = cell_coord(sp.x, G.lo[0], G.inv_x, G.dim[0]);
    const int iy = cell_coord(sp.y, G.lo[1], G.inv_cell, G.dim[1]);
    const int iz = cell_coord(sp.z, G.lo[2], G.inv_cell, G.dim[2]);
    return ix + G.dim[0] * (iy + G.dim[1] * iz);
}

// Bounding sphere of pill g into P.spheres, folded into this thread's running bounds
// (the radius by its size: contacts squeeze radii past zero, and spheres_overlap squares
// the sum, so the search's reach is that of the largest size).
__device__ __forceinline__ void bound_pill(const Params &P, int g, float mn[3], float mx[3], float &mr)
{
    const float4 sp = bp_sphere(P, g);
    P.spheres[g] = sp;
    mn[0] = fminf(mn[0], sp.x); mn[1] = fminf(mn[1], sp.y); mn[2] = fminf(mn[2], sp.z);
    mx[0] = fmaxf(mx[0], sp.x); mx[1] = fmaxf(mx[1], sp.y); mx[2] = fmaxf(mx[2], sp.z);
    mr = fmaxf(mr, fabsf(sp.w));
}

// Warp-wide min/max of the running bounds, merged into `bounds` by lane 0:
// bounds[0..2] = enc(-min c), bounds[3..5] = enc(max c), bounds[6] = enc(max |R|),
// all zero before the first merge.  Every lane of the warp must call it.
__device__ __forceinline__ void merge_bounds_to(unsigned int *bounds, float mn[3], float mx[3], float mr)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        for (int c = 0; c < 3; ++c) {
            mn[c] = fminf(mn[c], __shfl_xor_sync(0xffffffffu, mn[c], o));
            mx[c] = fmaxf(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], o));
        }
        mr = fmaxf(mr, __shfl_xor_sync(0xffffffffu, mr, o));
    }
    if ((threadIdx.x & 31) == 0 && mr > 0.f) {
        for (int c = 0; c < 3; ++c) {
            atomicMax(bounds + c, ord_enc(-mn[c]));
            atomicMax(bounds + 3 + c, ord_enc(mx[c]));
        }
        atomicMax(bounds + 6, ord_enc(mr));
    }
}

__device__ __forceinline__ void merge_bounds(const Params &P, float mn[3], float mx[3], float mr)
{
    merge_bounds_to(P.bounds, mn, mx, mr);
}

// ---------------------------------------------------------------- oversized pills
// One pill far longer than the rest (a segment stretched by an impact) would
// set the cell of the whole grid through the largest bounding radius and put
// thousands of pills in each cell.  The multi-kernel broadphase therefore
// histograms the radii (16 bins per octave: the float's exponent and top four
// mantissa bits) and sizes the cell for the cut radius below which all but at
// most big_cap pills lie (the cluster's grid does the same).  The pills above it sit in the cells like the others
// but are paired from their own side (emit_big).  The pair set is unchanged:
// every candidate is still decided by spheres_overlap.
constexpr unsigned int kRadBinBase = (127u - 20u) << 4;  // bin 0 starts at 2^-20
__device__ __forceinline__ int rad_bin(float R)
{
    const int b = (int)(__float_as_uint(R) >> 19) - (int)kRadBinBase;
    return min(max(b, 0), kRadBins - 1);
}
// Upper edge of bin b (exclusive): every radius of bins <= b is below it.
__device__ __forceinline__ float rad_bin_top(int b) { return __uint_as_float(((unsigned)b + 1u + kRadBinBase) << 19); }

// Oversized pills are those with rad_bin(R) > b_cut: the bits of R, as an
// unsigned number, above this threshold (none when b_cut is the last bin).
__device__ __forceinline__ unsigned int big_threshold(int b_cut)
{
    return b_cut < kRadBins - 1 ? (((unsigned)b_cut + 1u + kRadBinBase) << 19) - 1u : 0xffffffffu;
}

// Cut bin from the histogram, by every thread of a block of kRadBins / PER
// threads (the same result in every block): the smallest b such that bins above
// b hold at most `cap` pills, or all / `share` of those counted if that is fewer
// (a cut that takes half of a few pills out makes cells far below their size).  Returns b_cut; *r_cut = the top edge of bin
// b_cut, or the largest radius when no pill lies above it.  sh: kRadBins + 33
// ints of shared memory.
template <int PER>
__device__ __forceinline__ int choose_cut(const int *hist, int cap, int share, float r_max, int *sh, float *r_cut)
{
    int *h = sh, *ws = sh + kRadBins;
    const int b0 = kRadBins - 1 - PER * threadIdx.x;  // bins b0, b0 - 1, ... (suffix sums from the top)
    int n[PER], tot, sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) sum += n[j] = hist[b0 - j];
    int above = block_excl_scan(sum, ws, &tot);  // pills in bins > b0
    cap = min(cap, tot / share);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        h[b0 - j] = above;
        above += n[j];
    }
    __syncthreads();
    // bins b with (pills above b) <= cap form a top range [b_cut, kRadBins); its size
    int n_ok = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) n_ok += __syncthreads_count(h[b0 - j] <= cap);
    const int b_cut = max(kRadBins - n_ok, 0);
    const bool none_above = h[b_cut] == 0;
    __syncthreads();
    *r_cut = none_above ? r_max : rad_bin_top(b_cut);
    return none_above ? kRadBins - 1 : b_cut;
}

// One more pill of radius R in the histogram; the lanes `act` call it together
// (most pills of a scene share a few bins: one addition per bin and warp).
__device__ __forceinline__ void hist_add(int *hist, unsigned act, float R)
{
    const int bin = rad_bin(R);
    const unsigned peers = __match_any_sync(act, bin);
    if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(hist + bin, __popc(peers));
}

__device__ __forceinline__ void count_pill(const Params &P, const Grid &G, int g)
{
    const int cell = bp_cell(G, P.spheres[g]);
    P.cell_of[g] = cell;
    atomicAdd(P.cell_count + cell, 1);
}

// Places pill g in its cell (entries from `first`, the cell's start), with a
// copy of its bounding sphere and group in cell order for the pair search,
// and returns the cell's count towards zero, ready for the next substep.
__device__ __forceinline__ void scatter_pill(const Params &P, int g, int cell, int first)
{
    const int pos = first + atomicSub(P.cell_count + cell, 1) - 1;
    P.cell_pills[pos] = g;
    P.cell_sph[pos] = P.spheres[g];
    P.cell_grp[pos] = P.seg_group[g];
}

// Candidate pairs between one grid cell and one of its neighbours, by one
// warp (the frame solver's search).  Every pair of pills whose cells are neighbours is visited exactly
// once: from the lower cell of the 13 "forward" neighbour offsets (dz = 1;
// dz = 0, dy = 1; dz = dy = 0, dx = 1), and inside one cell from the pill at
// the lower position.  Work unit u = 14 c + k pairs cell c with its forward
// neighbour k < 13, or with itself (k = 13), so that the work of a crowded
// neighbourhood is spread over 14 warps.  The cell's pills sit one per lane
// (32 at a time); the neighbour's pills are loaded 32 at a time from the
// cell-order sphere / group copies (coalesced) and broadcast to all lanes,
// so each step tests up to 32 pairs.  Hits are compacted with a ballot and
// their output slots reserved with one atomic per step; pairs are written as
// (lower id, higher id).  start(c) is the first entry of cell c in cell
// order (start(c + 1) its end).
constexpr int kEmitUnits = 14;

template <int STEP, class StartFn>
__device__ __forceinline__ void emit_cell(const Params &P, const Grid &G, int u, StartFn start)
{
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int c = u / kEmitUnits, k = u % kEmitUnits;
    const int c0 = start(c), c1 = start(c + 1);
    if (c0 >= c1) return;  // empty cell (uniform over the warp)
    int d = c;
    if (k < 13) {
        int dx, dy, dz;
        if (k < 9) {
            dx = k % 3 - 1; dy = k / 3 - 1; dz = 1;
        } else if (k < 12) {
            dx = k - 10; dy = 1; dz = 0;
        } else {
            dx = 1; dy = 0; dz = 0;
        }
        const int ix = c % G.dim[0], iy = (c / G.dim[0]) % G.dim[1], iz = c / (G.dim[0] * G.dim[1]);
        const int x = ix + dx, y = iy + dy, z = iz + dz;
        if (x < 0 || x >= G.dim[0] || y < 0 || y >= G.dim[1] || z >= G.dim[2]) return;
        d = x + G.dim[0] * (y + G.dim[1] * z);
    }
    const int d0 = start(d), d1 = start(d + 1);
    if (d0 >= d1) return;
    for (int ob = c0; ob < c1; ob += 32) {
        const int pa = ob + lane;
        const bool own = pa < c1;
        const float4 sa = own ? P.cell_sph[pa] : make_float4(0.f, 0.f, 0.f, 0.f);
        const int ga = own ? P.cell_grp[pa] : 0;
        // inside the own cell only pairs with pb > pa: candidates from this chunk on
        for (int cb = (k == 13 ? ob : d0); cb < d1; cb += 32) {
            const int q = cb + lane;
            float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);
            int cg = 0;
            if (q < d1) {
                cs = P.cell_sph[q];
                cg = P.cell_grp[q];
            }
            const int m = min(32, d1 - cb);
            // STEP candidates per step: their broadcasts and tests are independent
            for (int j0 = 0; j0 < m; j0 += STEP) {
                bool hit[STEP];
#pragma unroll
                for (int t = 0; t < STEP; ++t) {
                    const int j = j0 + t;  // past m: no candidate (j & 31 is still a valid source lane)
                    float4 sj;
                    sj.x = __shfl_sync(full, cs.x, j & 31);
                    sj.y = __shfl_sync(full, cs.y, j & 31);
                    sj.z = __shfl_sync(full, cs.z, j & 31);
                    sj.w = __shfl_sync(full, cs.w, j & 31);
                    const int gj = __shfl_sync(full, cg, j & 31);
                    hit[t] = j < m && own && cb + j > pa && gj != ga && spheres_overlap(sa, sj);
                }
#pragma unroll
                for (int t = 0; t < STEP; ++t) {
                    const unsigned hm = __ballot_sync(full, hit[t]);
                    if (hm) {
                        int out = 0;
                        if (lane == 0) out = atomicAdd(P.npairs, __popc(hm));
                        out = __shfl_sync(full, out, 0);
                        if (hit[t]) {
                            const int idx = out + __popc(hm & ((1u << lane) - 1u));
                            if (idx < P.max_pairs) {
                                const int a = P.cell_pills[pa], b = P.cell_pills[cb + j0 + t];
                                P.pairs[idx] = make_int2(min(a, b), max(a, b));
                                if (P.pair_v) P.pair_v[idx] = make_int2(P.seg_v0[min(a, b)], P.seg_v0[max(a, b)]);
                                if (P.lam_pair) P.lam_pair[idx] = 0.f;
                            }
                        }
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------- pair search of large scenes
// Hits wait in the warp's shared buffer as cell-order entries: kLanePairs a
// lane, rows one word apart modulo the banks, so that appending (a row per
// lane) and flushing (along rows) are both free of bank conflicts.
constexpr int kLanePairs = 24, kLaneRow = kLanePairs + 1, kEmitBuf = 32 * kLaneRow;

// Writes pair number idx of pills (a, first vertex va) and (b, vb) as (lower id, higher id).
__device__ __forceinline__ void put_pair(const Params &P, int idx, int a, int va, int b, int vb)
{
    if (idx >= P.max_pairs) return;
    if (P.pairs) P.pairs[idx] = make_int2(min(a, b), max(a, b));
    if (P.pair_v) P.pair_v[idx] = a < b ? make_int2(va, vb) : make_int2(vb, va);
    if (P.lam_pair) P.lam_pair[idx] = 0.f;
}

// Flushes the lanes' rows (cnt hits in this lane's, found for pill ia with
// first vertex va) with one atomic and coalesced stores, row after row: the
// pairs of one pill stay together in the list, so that lanes of the contact
// pass share its vertices.  Output t belongs to the last row that starts at or
// before t.  Every lane of the warp calls it.
__device__ __forceinline__ void flush_rows(const Params &P, const int *buf, int cnt, int ia, int va, int lane)
{
    const unsigned full = 0xffffffffu;
    const int inc = warp_incl_scan(cnt), off = inc - cnt;
    const int total = __shfl_sync(full, inc, 31);
    int base = 0;
    if (lane == 0) base = atomicAdd(P.npairs, total);
    base = __shfl_sync(full, base, 0);
    __syncwarp();
    for (int t0 = 0; t0 < total; t0 += 32) {
        const int t = min(t0 + lane, total - 1);
        int l = 0;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1)
            if (__shfl_sync(full, off, l + s) <= t) l += s;
        const int k = t - __shfl_sync(full, off, l);
        const int a = __shfl_sync(full, ia, l), v = __shfl_sync(full, va, l);
        if (t0 + lane < total) {
            const int b = P.cell_pills[buf[l * kLaneRow + k]];
            put_pair(P, base + t, a, v, b, P.pair_v ? P.seg_v0[b] : 0);
        }
    }
    __syncwarp();
}

// The row's hits of another group than ga, moved up; returns their number.  The
// groups are looked up for the hits only, four at a time: one candidate in ten is one.
__device__ __forceinline__ int other_groups(const Params &P, int *row, int cnt, int ga)
{
    int n = 0;
    for (int j = 0; j < cnt; j += 4) {
        int q[4], g[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            q[t] = j + t < cnt ? row[j + t] : -1;
            g[t] = q[t] >= 0 ? P.cell_grp[q[t]] : ga;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (g[t] != ga) row[n++] = q[t];
    }
    return n;
}

// spheres_overlap with the components in packed pairs (add and multiply two
// floats at a time, each rounded as the scalar operation): (b - a) and, in the
// fourth place, Ra + Rb, then their squares.  na = (-ax, -ay, -az, Ra).
__device__ __forceinline__ bool spheres_overlap2(float4 na, float4 b)
{
    float ex, ey, ez, rs;
    asm("{\n\t.reg .b64 p, q, r, s;\n\t"
        "mov.b64 p, {%4, %5};\n\tmov.b64 q, {%6, %7};\n\t"
        "mov.b64 r, {%8, %9};\n\tmov.b64 s, {%10, %11};\n\t"
        "add.rn.f32x2 p, p, r;\n\tadd.rn.f32x2 q, q, s;\n\t"
        "mul.rn.f32x2 p, p, p;\n\tmul.rn.f32x2 q, q, q;\n\t"
        "mov.b64 {%0, %1}, p;\n\tmov.b64 {%2, %3}, q;\n\t}"
        : "=f"(ex), "=f"(ey), "=f"(ez), "=f"(rs)
        : "f"(na.x), "f"(na.y), "f"(na.z), "f"(na.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w));
    return __fadd_rn(__fadd_rn(ex, ey), ez) <= rs;
}

// Candidate pairs of the n pills in the cells, up to the cut, L lanes per pill in cell order
// (a warp step takes entries p0 .. p0 + 32 / L - 1 of the cell-order copies).
// Each tests the pills of its own row after it and those of the four forward
// rows (dz = 1; dz = 0, dy = 1), within its reach along x (its own radius and the
// largest), so every pair that overlaps is tested once, from the pill that comes
// first.  Cells are numbered along x, so these are five runs of the cell order: what
// follows in the own row, and part of four others.  A pill's lanes walk its runs
// end to end, four candidates a lane and step; the warp takes the longest walk's
// number of steps.
// L = 1 where the pills fill the GPU: settled strands (300,000 pills, 8.8
// million pairs) took 216 us a search with the oversized pills when this walk was
// made, in cubic cells (211 candidates a pill; make_grid_from's thinner ones leave 159),
// against 469 us with fourteen lists each walked to the warp's longest and the
// oversized pills tested against their whole list.  More lanes shorten the walk where
// the pills do not fill the GPU.
template <int L>
__device__ __forceinline__ void emit_pills(const Params &P, const Grid &G, unsigned int big, int n, int warp,
                                           int nwarps, int *buf, int lane)
{
    const unsigned full = 0xffffffffu;
    constexpr int kPer = 32 / L;  // pills per warp step
    const int sub = lane % L;
    int *row = buf + lane * kLaneRow;
    for (int p0 = warp * kPer; p0 < n; p0 += nwarps * kPer) {
        const int p = p0 + lane / L;
        float4 na = make_float4(0.f, 0.f, 0.f, 0.f);
        int ga = 0, ia = 0, va = 0, cnt = 0;
        int q = 0, end = 0, q1 = 0, e1 = 0, q2 = 0, e2 = 0, q3 = 0, e3 = 0, q4 = 0, e4 = 0;
        if (p < n) {
            const float4 sa = P.cell_sph[p];
            if (!(__float_as_uint(sa.w) > big)) {
                na = make_float4(-sa.x, -sa.y, -sa.z, sa.w);
                ga = P.cell_grp[p];
                ia = P.cell_pills[p];
                const int iy = cell_coord(sa.y, G.lo[1], G.inv_cell, G.dim[1]);
                const int iz = cell_coord(sa.z, G.lo[2], G.inv_cell, G.dim[2]);
                int x0, x1;
                cell_range(sa.x, __fadd_rn(fabsf(sa.w), G.r_cut), G.lo[0], G.inv_x, G.dim[0], x0, x1);
                ++x1;
                const int r0 = G.dim[0] * (iy + G.dim[1] * iz), ry = G.dim[0], rz = G.dim[0] * G.dim[1];
                const int *cs = P.cell_start;
                const bool up = iy + 1 < G.dim[1], down = iy > 0, next = iz + 1 < G.dim[2];
                q = p + 1;
                end = cs[r0 + x1];
                if (up) { q1 = cs[r0 + ry + x0]; e1 = cs[r0 + ry + x1]; }
                if (next && down) { q2 = cs[r0 + rz - ry + x0]; e2 = cs[r0 + rz - ry + x1]; }
                if (next) { q3 = cs[r0 + rz + x0]; e3 = cs[r0 + rz + x1]; }
                if (next && up) { q4 = cs[r0 + rz + ry + x0]; e4 = cs[r0 + rz + ry + x1]; }
                if (P.pair_v) va = P.seg_v0[ia];
            }
        }
        int left = 4;  // runs after the current one
        while (true) {
            while (q >= end && left > 0) {
                q = q1; end = e1;
                q1 = q2; e1 = e2;
                q2 = q3; e2 = e3;
                q3 = q4; e3 = e4;
                --left;
            }
            if (!__any_sync(full, q < end)) break;
            float4 cs[4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (q + t * L + sub < end) cs[t] = P.cell_sph[q + t * L + sub];
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (q + t * L + sub < end && spheres_overlap2(na, cs[t]) && !(__float_as_uint(cs[t].w) > big))
                    row[cnt++] = q + t * L + sub;
            q += 4 * L;
            if (__any_sync(full, cnt > kLanePairs - 4)) {
                cnt = other_groups(P, row, cnt, ga);
                flush_rows(P, buf, cnt, ia, va, lane);
                cnt = 0;
            }
        }
        cnt = other_groups(P, row, cnt, ga);
        if (__any_sync(full, cnt > 0)) flush_rows(P, buf, cnt, ia, va, lane);
    }
}

__device__ __forceinline__ void flush_big(const Params &P, const int *buf, int cnt, int ia, int va, int lane)
{
    int base = 0;
    if (lane == 0) base = atomicAdd(P.npairs, cnt);
    base = __shfl_sync(0xffffffffu, base, 0);
    __syncwarp();
    for (int t = lane; t < cnt; t += 32) {
        const int b = P.cell_pills[buf[t]];
        put_pair(P, base + t, ia, va, b, P.pair_v ? P.seg_v0[b] : 0);
    }
    __syncwarp();
}

// Candidate pairs of oversized pill i of the list, by one warp: all pills up to
// the cut, and of the oversized ones those that come after it in the order of
// descending radius (equal radii by id), so that each pair is found once, from
// its larger pill, and lies within |Ri| + max(|Ri|, r_cut) of its centre.  The
// cells of that box (cell_range) are rows
// of the cell order; 32 rows' ends are loaded at a time.  (Radii can be
// negative: contacts squeeze them past zero; their bits then sort above every
// cut.)
__device__ __forceinline__ void emit_big(const Params &P, const Grid &G, unsigned int big, int i, int *buf, int lane)
{
    const unsigned full = 0xffffffffu;
    const int gi = P.big_list[i];
    const float4 si = P.spheres[gi];
    const float4 na = make_float4(-si.x, -si.y, -si.z, si.w);
    const float Ri = fabsf(si.w);
    const int grp = P.seg_group[gi], vi = P.pair_v ? P.seg_v0[gi] : 0;
    const float reach = __fadd_rn(Ri, fmaxf(Ri, G.r_cut));
    const float c[3] = {si.x, si.y, si.z};
    int lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) cell_range(c[k], reach, G.lo[k], k ? G.inv_cell : G.inv_x, G.dim[k], lo[k], hi[k]);
    const int ny = hi[1] - lo[1] + 1, rows = ny * (hi[2] - lo[2] + 1);
    int cnt = 0;  // hits in buf (uniform over the warp)
    for (int rb = 0; rb < rows; rb += 32) {
        int s0 = 0, s1 = 0;
        if (rb + lane < rows) {
            const int y = lo[1] + (rb + lane) % ny, z = lo[2] + (rb + lane) / ny;
            const int row = G.dim[0] * (y + G.dim[1] * z);
            s0 = P.cell_start[row + lo[0]];
            s1 = P.cell_start[row + hi[0] + 1];
        }
        const int nr = min(32, rows - rb);
        for (int r = 0; r < nr; ++r) {
            const int p0 = __shfl_sync(full, s0, r), p1 = __shfl_sync(full, s1, r);
            for (int pb = p0; pb < p1; pb += 32) {
                const int q = pb + lane;
                bool hit = false;
                if (q < p1) {
                    const float4 sj = P.cell_sph[q];
                    hit = P.cell_grp[q] != grp && spheres_overlap2(na, sj);
                    if (hit && __float_as_uint(sj.w) > big) {
                        const float Rj = fabsf(sj.w);
                        hit = Rj < Ri || (Rj == Ri && P.cell_pills[q] < gi);
                    }
                }
                const unsigned m = __ballot_sync(full, hit);
                if (hit) buf[cnt + __popc(m & ((1u << lane) - 1u))] = q;
                cnt += __popc(m);
                if (cnt > kEmitBuf - 32) {
                    __syncwarp();
                    flush_big(P, buf, cnt, gi, vi, lane);
                    cnt = 0;
                }
            }
        }
    }
    __syncwarp();
    if (cnt) flush_big(P, buf, cnt, gi, vi, lane);
}

// ================================================================ contacts
// Correction of vertex v: position d, radius dr (= scale change x rest radius).
__device__ __forceinline__ void acc_add(const Params &P, int v, V3 d, float dr)
{
    unsigned long long *a = P.acc + 2 * (size_t)v;
    atomicAdd(a + 0, fix_pack(d.x, d.y, P.fix_scale));
    atomicAdd(a + 1, fix_pack(d.z, dr, P.fix_scale));
    atomicAdd(P.cnt + v, 1);
}

__device__ __forceinline__ float4 world_of(const Params &P, int v)
{
    float4 x = P.X[v], o = P.rod_origin[P.rod_of_v[v]];
    return make_float4(__fadd_rn(x.x, o.x), __fadd_rn(x.y, o.y), __fadd_rn(x.z, o.z), x.w);
}


// Pill-pill contacts (Sec. 7.2): narrowphase on the current state, then one
// XPBD update of pair i's multiplier if the pills interpenetrate.
struct ContactPair {
    PillPair Q;
    int vs[4];      // the pills' vertices a1, a2, b1, b2
    float rbar[4];  // their rest radii
};

// World positions and radii packed by the preceding sweep: the pair's first
// vertices pv and four 16-byte gathers (rest radii: only if active).
__device__ __forceinline__ void contact_load_packed(const Params &P, int2 pv, ContactPair &c)
{
    const float4 xa1 = P.XW[pv.x], xa2 = P.XW[pv.x + 1], xb1 = P.XW[pv.y], xb2 = P.XW[pv.y + 1];
    c.vs[0] = pv.x; c.vs[1] = pv.x + 1; c.vs[2] = pv.y; c.vs[3] = pv.y + 1;
    c.Q.a1 = xyz(xa1); c.Q.a2 = xyz(xa2); c.Q.b1 = xyz(xb1); c.Q.b2 = xyz(xb2);
    c.Q.ra1 = xa1.w; c.Q.ra2 = xa2.w; c.Q.rb1 = xb1.w; c.Q.rb2 = xb2.w;
}

__device__ __forceinline__ void contact_load(const Params &P, int i, ContactPair &c)
{
    if (P.XW) {
        contact_load_packed(P, P.pair_v[i], c);
        return;
    }
    const int2 pr = P.pairs[i];
    // the segments' first vertices, stored beside the pair by the pair search
    // (one dependent load less on the contact pass's chain)
    const int2 pv = P.pair_v ? P.pair_v[i] : make_int2(P.seg_v0[pr.x], P.seg_v0[pr.y]);
    const int va = pv.x, vb = pv.y;
    // the segments' rod origins, loaded beside their first vertices (not through rod_of_v)
    const float4 oa = P.seg_org[pr.x], ob = P.seg_org[pr.y];
    auto wpos = [&](int v, const float4 &o) {
        const float4 x = P.X[v];
        return make_float4(__fadd_rn(x.x, o.x), __fadd_rn(x.y, o.y), __fadd_rn(x.z, o.z), x.w);
    };
    const float4 xa1 = wpos(va, oa), xa2 = wpos(va + 1, oa), xb1 = wpos(vb, ob), xb2 = wpos(vb + 1, ob);
    c.vs[0] = va; c.vs[1] = va + 1; c.vs[2] = vb; c.vs[3] = vb + 1;
    c.rbar[0] = P.RV0[va].w; c.rbar[1] = P.RV0[va + 1].w; c.rbar[2] = P.RV0[vb].w; c.rbar[3] = P.RV0[vb + 1].w;
    c.Q.a1 = xyz(xa1); c.Q.a2 = xyz(xa2); c.Q.b1 = xyz(xb1); c.Q.b2 = xyz(xb2);
    c.Q.ra1 = __fmul_rn(xa1.w, c.rbar[0]); c.Q.ra2 = __fmul_rn(xa2.w, c.rbar[1]);
    c.Q.rb1 = __fmul_rn(xb1.w, c.rbar[2]); c.Q.rb2 = __fmul_rn(xb2.w, c.rbar[3]);
}

// The update of pair i at contact parameter al; vertices t0, t0 + tstep, ...
// of the four are accumulated by this thread, and the multiplier is stored if
// write_lam.  With `warp` all 32 lanes handle the same pair (the early return
// is uniform) and the multiplier is written only after every lane has read it.
// What the update of pair i reads besides the pair's geometry: the four
// vertices' rest radii, inverse masses and scale weights, and its multiplier.
struct ApplyData {
    float rbar[4], wx[4], wsv[4], lam;
};

__device__ __forceinline__ void apply_data(const Params &P, int i, const ContactPair &c, ApplyData &D)
{
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float4 m = P.CM[c.vs[t]];  // rest radius, inverse mass, scale weight
        D.rbar[t] = P.XW ? m.x : c.rbar[t];
        D.wx[t] = m.y;
        D.wsv[t] = m.z;
    }
    D.lam = P.lam_pair[i];
}

__device__ __forceinline__ bool contact_apply(const Params &P, int i, float at, const ContactPair &c, float al, int t0,
                                              int tstep, bool write_lam, bool warp)
{
    float be;
    const float C = coll_f(c.Q, al, be);
    V3 d = lerp3(c.Q.a1, c.Q.a2, al) - lerp3(c.Q.b1, c.Q.b2, be);
    float dist = sqrtf(dot(d, d));
    if (!(C < 0.f) || dist < 1e-12f) return false;
    V3 n = (1.f / dist) * d;
    ApplyData D;  // loaded only for an active pair
    apply_data(P, i, c, D);
    const float wt[4] = {1.f - al, al, -(1.f - be), -be};
    float den = at;
#pragma unroll
    for (int t = 0; t < 4; ++t)
        den += D.wx[t] * wt[t] * wt[t] + D.wsv[t] * wt[t] * wt[t] * D.rbar[t] * D.rbar[t];
    const float dl = (-C - at * D.lam) / den;
    if (warp) __syncwarp();
    if (write_lam) P.lam_pair[i] = D.lam + dl;
#pragma unroll
    for (int t = 0; t < 4; ++t)
        if (t >= t0 && (t - t0) % tstep == 0)
            acc_add(P, c.vs[t], (D.wx[t] * wt[t] * dl) * n, -D.wsv[t] * fabsf(wt[t]) * D.rbar[t] * dl * D.rbar[t]);
    return true;
}

// Certified early-out of the narrowphase.  Every probe of the search
// evaluates C = |pa - pb| - ra - rb >= D - max(ra) - max(rb), D the distance
// of the two axis segments, and for any direction n, D is at least the gap
// between the segments' projections on n:
//   gap(n) |n| = |n.e| - (|n.da| + |n.db|) / 2,   e = ma - mb (midpoints).
// When gap(n) exceeds the larger radius of each pill by a margin (1e-3 of the
// radii plus 1e-5 of the coordinates' magnitude, far above the FP32 rounding
// of either computation), the search could only find C > 0: the pair is
// inactive and skipping it changes no result.  Two directions are tried: the
// line through the midpoints, then the direction between the closest points
// of the axes (clamped closed form; its rounding only loosens the bound).
// Returns false when either certifies the pair inactive.
__device__ __forceinline__ bool sat_separated(V3 n, V3 e, V3 da, V3 db, float lim)
{
    const float nn = dot(n, n);
    return nn > 0.f && fabsf(dot(n, e)) - 0.5f * (fabsf(dot(n, da)) + fabsf(dot(n, db))) > lim * sqrtf(nn);
}

__device__ __forceinline__ bool contact_may_touch(const PillPair &Q)
{
    const V3 ma = 0.5f * (Q.a1 + Q.a2), mb = 0.5f * (Q.b1 + Q.b2);
    const V3 e = ma - mb, da = Q.a2 - Q.a1, db = Q.b2 - Q.b1;
    const float rho = fmaxf(Q.ra1, Q.ra2) + fmaxf(Q.rb1, Q.rb2);
    const float mag = fmaxf(fmaxf(fmaxf(fabsf(ma.x), fabsf(ma.y)), fmaxf(fabsf(ma.z), fabsf(mb.x))),
                            fmaxf(fabsf(mb.y), fabsf(mb.z)));
    const float lim = rho + 1e-3f * rho + 1e-5f * mag;
    if (sat_separated(e, e, da, db, lim)) return false;
    // closest points a1 + s da, b1 + t db of the two axes, s, t in [0, 1]
    const V3 r = Q.a1 - Q.b1;
    const float a = dot(da, da), b = dot(da, db), c = dot(da, r), ee = dot(db, db), f = dot(db, r);
    if (!(a > 0.f) || !(ee > 0.f)) return true;
    const float den = a * ee - b * b;
    float sp = den > 1e-6f * a * ee ? fminf(fmaxf((b * f - c * ee) / den, 0.f), 1.f) : 0.f;
    float tq = (b * sp + f) / ee;
    if (tq < 0.f) {
        tq = 0.f;
        sp = fminf(fmaxf(-c / a, 0.f), 1.f);
    } else if (tq > 1.f) {
        tq = 1.f;
        sp = fminf(fmaxf((b - c) / a, 0.f), 1.f);
    }
    const V3 n = (Q.a1 + sp * da) - (Q.b1 + tq * db);
    return !sat_separated(n, e, da, db, lim);
}

// The same certificate from the pills' packs (pill_box), for the pass over many
// pairs: with e the line through the midpoints, the closest points e + s da - t db,
// s, t in [-1/2, 1/2], by alternating clamped minima (approximate divisions: any
// direction n gives a valid bound, and the padding covers the bound's own
// rounding; a NaN or infinite n certifies nothing).  One 256-bit load per
// pill and about 65 operations; from the four vertices, with IEEE divisions and
// square roots, the test took 350 instructions a warp.
__device__ __forceinline__ bool boxes_may_touch(const Params &P, int2 pv)
{
    float4 am, ad, bm, bd;
    ld_record(P.PB + 2 * (size_t)pv.x, am, ad);
    ld_record(P.PB + 2 * (size_t)pv.y, bm, bd);
    const V3 e = xyz(am) - xyz(bm), da = xyz(ad), db = xyz(bd);
    const float lim = am.w + bm.w;
    const float ee = dot(e, e), ea = dot(e, da), eb = dot(e, db);
    if (ee - 0.5f * (fabsf(ea) + fabsf(eb)) > lim * sqrt_approx(ee)) return false;
    const float ab = dot(da, db);
    const float den = ad.w * bd.w - ab * ab;
    const float s0 = den > 1e-6f * ad.w * bd.w ? fminf(fmaxf(fdiv(ab * eb - bd.w * ea, den), -0.5f), 0.5f) : 0.f;
    const float t = fminf(fmaxf(fdiv(ab * s0 + eb, bd.w), -0.5f), 0.5f);
    const float s = fminf(fmaxf(fdiv(ab * t - ea, ad.w), -0.5f), 0.5f);
    const V3 n = e + s * da - t * db;
    const float gap = fabsf(dot(n, e)) - 0.5f * (fabsf(dot(n, da)) + fabsf(dot(n, db)));
    return !(gap > lim * sqrt_approx(dot(n, n)));
}

// Pair i by one thread.
__device__ __forceinline__ void contact_pair(const Params &P, int i, float at)
{
    ContactPair c;
    contact_load(P, i, c);
    if (!contact_may_touch(c.Q)) return;
    pill_pair_axis(c.Q);
    contact_apply(P, i, at, c, dichotomous(c.Q), 0, 1, true, false);
}

// Pair i by one warp (all lanes call): the search four steps per round
// (dichotomous_warp), lane t < 4 accumulates vertex t, lane 0 stores the
// multiplier.  Same result as contact_pair, bit for bit.  Returns 0 (skipped
// by the early-out), 1 (searched) or 3 (searched, constraint active).
__device__ __forceinline__ int contact_pair_warp(const Params &P, int i, float at, int lane)
{
    ContactPair c;
    contact_load(P, i, c);
    if (!contact_may_touch(c.Q)) return 0;  // uniform over the warp
    pill_pair_axis(c.Q);
    const float al = dichotomous_warp(c.Q, lane);
    return contact_apply(P, i, at, c, al, lane, 4, lane == 0, true) ? 3 : 1;
}

// Pairs [0, np) a thread each, by the calling warp from chunk `chunk` of 32
// pairs on, every `stride`-th chunk.  The pairs that may touch are queued in
// the warp's buffer q (64 pairs of shared memory) and searched 32 at a time,
// so that the search runs on full warps however sparse the touching pairs are.
// The next chunk's pairs are loaded before this one is tested.  Same results
// as contact_pair.  Returns the warp's counts (searched, active), the same in
// every lane.
struct QueuedPair {
    int i;
    int2 v;
};

__device__ __forceinline__ bool queued_contact(const Params &P, QueuedPair j, float at)
{
    ContactPair c;
    if (P.XW)
        contact_load_packed(P, j.v, c);
    else
        contact_load(P, j.i, c);
    pill_pair_axis(c.Q);
    return contact_apply(P, j.i, at, c, dichotomous_packed(c.Q), 0, 1, true, false);
}

__device__ __forceinline__ int2 contact_pairs_compacted(const Params &P, int np, float at, int chunk, int stride,
                                                        QueuedPair *q, int lane)
{
    const unsigned full = 0xffffffffu;
    int qn = 0;  // queued pairs (uniform over the warp)
    int2 counts = make_int2(0, 0);
    int i = chunk * 32 + lane;
    int2 next = i < np ? P.pair_v[i] : make_int2(0, 0);
    for (int base = chunk * 32; base < np; base += stride * 32) {
        const int2 pv = next;
        i = base + lane;
        const int ahead = i + stride * 32;
        if (ahead < np) next = P.pair_v[ahead];
        bool maybe = false;
        if (i < np) {
            if (P.PB) {
                maybe = boxes_may_touch(P, pv);
            } else {
                ContactPair c;
                contact_load(P, i, c);
                maybe = contact_may_touch(c.Q);
            }
        }
        const unsigned m = __ballot_sync(full, maybe);
        if (maybe) q[qn + __popc(m & ((1u << lane) - 1u))] = QueuedPair{i, pv};
        qn += __popc(m);
        __syncwarp();
        if (qn >= 32) {
            const bool act = queued_contact(P, q[lane], at);
            counts.x += 32;
            counts.y += __popc(__ballot_sync(full, act));
            __syncwarp();
            qn -= 32;
            if (lane < qn) q[lane] = q[lane + 32];
            __syncwarp();
        }
    }
    const bool act = lane < qn && queued_contact(P, q[lane], at);
    counts.x += qn;
    counts.y += __popc(__ballot_sync(full, act));
    __syncwarp();
    return counts;
}

// Half-plane constraints of vertex v's sphere (Sec. 7).
__device__ __forceinline__ void contact_planes(const Params &P, int v, float at)
{
    const float4 x = world_of(P, v);
    const float rbar = P.RV0[v].w;
    const float4 m = P.RV1[v];
    const float w = inv_mass(m);
    for (int k = 0; k < P.n_planes; ++k) {
        const float4 pl = P.planes[k];
        const float C = pl.x * x.x + pl.y * x.y + pl.z * x.z - pl.w - x.w * rbar;
        if (!(C < 0.f)) continue;
        float *lp = P.lam_plane + (size_t)v * P.n_planes + k;
        const float den = w + m.y * rbar * rbar + at;
        const float dl = (-C - at * *lp) / den;
        *lp += dl;
        acc_add(P, v, (w * dl) * v3(pl.x, pl.y, pl.z), -m.y * rbar * dl * rbar);
    }
}

// ================================================================ bundles
// Rotation maximising trace(R^T A) (A row-major 3x3) by the iterative
// rotation extraction of Mueller et al. 2016 ("A Robust Method to Extract the
// Rotational Part of Deformations"): with r_k, a_k the columns of R(q) and A,
// turn q by the axis-angle w = sum_k r_k x a_k / (|sum_k r_k . a_k| + eps)
// until the step vanishes.  Starts from q0 (the method converges in a few
// steps from a start near the answer; from far away, e.g. the identity
// against a half turn, it needs many).  *converged is false when the 32-step
// cap is reached with a step above 1e-5 rad.
__device__ __forceinline__ float4 extract_rotation(const float *A, float4 q0, bool *converged)
{
    float4 q = q0;
    bool done = false;
#pragma unroll 1
    for (int it = 0; it < 32; ++it) {
        const V3 r0 = qrot(q, v3(1.f, 0.f, 0.f)), r1 = qrot(q, v3(0.f, 1.f, 0.f)), r2 = qrot(q, v3(0.f, 0.f, 1.f));
        const V3 a0 = v3(A[0], A[3], A[6]), a1 = v3(A[1], A[4], A[7]), a2 = v3(A[2], A[5], A[8]);
        const V3 num = cross(r0, a0) + cross(r1, a1) + cross(r2, a2);
        const float den = fabsf(dot(r0, a0) + dot(r1, a1) + dot(r2, a2)) + 1e-20f;
        const V3 w = (1.f / den) * num;
        const float ang = sqrtf(dot(w, w));
        if (!(ang > 1e-7f)) {
            done = true;
            break;
        }
        const float sh = sinf(0.5f * ang) / ang;
        q = qnormalize(qmul(make_float4(sh * w.x, sh * w.y, sh * w.z, cosf(0.5f * ang)), q));
        if (it == 31) done = ang <= 1e-5f;
    }
    *converged = done;
    return q;
}

// Shape matching of bundle cross-section c (Sec. 7.3) by one warp, member i
// on lane i (at most 32): T_i = [s_i R_i, c_i] (world position, scale, frame),
// A = sum_i [s_i R_i, c_i - mu][R_bar_i, c_bar_i - mu_bar]^T (warp sums),
// R* = argmax trace(R^T A), s* = <R*, A> / sum_i |B_bar_i|^2, then
// c_i = mu + s* R* (c_bar_i - mu_bar), s_i = s*, frame R* R_bar_i.  The
// member's pending contact corrections are applied first.
__device__ __forceinline__ void match_cross_section(const Params &P, int c)
{
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int o0 = P.xs_off[c], m = P.xs_off[c + 1] - o0;
    const bool mine = lane < m;
    int v = 0, g = -1;
    float4 x = make_float4(0.f, 0.f, 0.f, 1.f), org = x, rel = make_float4(0.f, 0.f, 0.f, 0.f), qb = org, q = org;
    if (mine) {
        v = P.xs_vert[o0 + lane];
        g = P.xs_seg[o0 + lane];
        x = apply_pending(P, v, P.X[v]);
        org = P.rod_origin[P.rod_of_v[v]];
        rel = P.xs_rel[o0 + lane];
        qb = P.xs_qbar[o0 + lane];
        if (g >= 0) q = P.Q[g];
    }
    const V3 cw = mine ? xyz(x) + xyz(org) : v3(0.f, 0.f, 0.f);
    V3 mu = cw;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mu.x += __shfl_xor_sync(full, mu.x, o);
        mu.y += __shfl_xor_sync(full, mu.y, o);
        mu.z += __shfl_xor_sync(full, mu.z, o);
    }
    mu = (1.f / m) * mu;
    float A[9];
    {
        const V3 d = cw - mu;
        const V3 rb = xyz(rel);
        const float dd[3] = {d.x, d.y, d.z}, bb[3] = {rb.x, rb.y, rb.z};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) A[3 * a + b] = mine ? dd[a] * bb[b] : 0.f;
        if (mine && g >= 0) {  // s R R_bar^T, column by column
            const V3 e[3] = {v3(1.f, 0.f, 0.f), v3(0.f, 1.f, 0.f), v3(0.f, 0.f, 1.f)};
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                // column b of R R_bar^T = R (R_bar^T e_b)
                const V3 col = qrot(q, qrot(qconj(qb), e[b]));
                A[b] += x.w * col.x;
                A[3 + b] += x.w * col.y;
                A[6 + b] += x.w * col.z;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) A[k] += __shfl_xor_sync(full, A[k], o);
    // start from the frame rotation R R_bar^T of the first member with a frame
    // segment (the members' frames turn with the cross-section)
    const unsigned framed = __ballot_sync(full, mine && g >= 0);
    float4 q0 = make_float4(0.f, 0.f, 0.f, 1.f);
    if (framed) {
        const int src = __ffs(framed) - 1;
        const float4 qq = qnormalize(qmul(q, qconj(qb)));
        q0 = make_float4(__shfl_sync(full, qq.x, src), __shfl_sync(full, qq.y, src), __shfl_sync(full, qq.z, src),
                         __shfl_sync(full, qq.w, src));
    }
    bool converged;
    const float4 qs = extract_rotation(A, q0, &converged);
    if (!converged && lane == 0) atomicOr(P.err, ERR_NOCONV);
    const V3 r0 = qrot(qs, v3(1.f, 0.f, 0.f)), r1 = qrot(qs, v3(0.f, 1.f, 0.f)), r2 = qrot(qs, v3(0.f, 0.f, 1.f));
    const float num = r0.x * A[0] + r0.y * A[3] + r0.z * A[6] + r1.x * A[1] + r1.y * A[4] + r1.z * A[7] +
                      r2.x * A[2] + r2.y * A[5] + r2.z * A[8];
    const float ss = num / P.xs_mub[c].w;
    if (mine) {
        const V3 cn = mu + ss * qrot(qs, xyz(rel));
        P.X[v] = make_float4(cn.x - org.x, cn.y - org.y, cn.z - org.z, ss);
        if (g >= 0) P.Q[g] = qnormalize(qmul(qs, qb));
    }
}

// ================================================================ skinning
// LBS frame of segment g (Sec. 7.4): the 3x4 similarity T_j Tbar_j^-1 =
// [s_m R_j Rbar_j^T | c_m - s_m R_j Rbar_j^T cbar_m] in world coordinates,
// stored as three float4 rows at the caller's segment id sperm[g].
constexpr int kLbsFrame = 2;  // float4 per skinning frame
__device__ __forceinline__ void lbs_frame_at(const Params &P, const float4 *__restrict__ LQ,
                                             const float4 *__restrict__ LC, const int *__restrict__ sperm,
                                             float4 *__restrict__ frames, int g)
{
    const int a = P.seg_v0[g];
    const float4 xa = P.X[a], xb = P.X[a + 1];
    const float sm = 0.5f * (xa.w + xb.w);
    const float4 q = P.Q[g], qb = LQ[g];
    const float4 r = qnormalize(qmul(q, qconj(qb)));  // R_j Rbar_j^T
    const float4 cb = LC[g];
    const V3 cm = 0.5f * (xyz(xa) + xyz(xb)) + xyz(P.rod_origin[P.rod_of_v[a]]);
    const V3 t = cm - sm * qrot(r, xyz(cb));
    float4 *f = frames + kLbsFrame * (size_t)sperm[g];
    f[0] = r;
    f[1] = make_float4(t.x, t.y, t.z, sm);
}

// Skinned position of mesh vertex i: sum_k w_k T_k Tbar_k^-1 rest_i over its
// four frames, from the vertex's rest position, frame ids and weights.  A
// frame is 32 bytes: the relative rotation r = R_j Rbar_j^T as a unit
// quaternion and (t, s_m) with t = c_m - s_m r cbar_m, so T Tbar^-1 p = s_m r p + t.
// Frame ids outside [0, ns) contribute nothing and raise the error word.
template <bool SHARED>
__device__ __forceinline__ float4 lbs_blend(float4 p, int4 id, float4 ww, int ns, const float4 *__restrict__ frames,
                                           int *err)
{
    const int ids[4] = {id.x, id.y, id.z, id.w};
    const float wv[4] = {ww.x, ww.y, ww.z, ww.w};
    float ox = 0.f, oy = 0.f, oz = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if ((unsigned)ids[k] >= (unsigned)ns) {
            atomicOr(err, ERR_OVERFLOW);
            continue;
        }
        float4 r, ts;
        if (SHARED) {  // a table of rotations, then one of translations (see lbs_gather_smem_kernel)
            r = frames[ids[k]];
            ts = frames[ns + ids[k]];
        } else {
            ld_record(frames + kLbsFrame * (size_t)ids[k], r, ts);
        }
        const V3 y = qrot(r, v3(p.x, p.y, p.z));
        ox += wv[k] * (ts.w * y.x + ts.x);
        oy += wv[k] * (ts.w * y.y + ts.y);
        oz += wv[k] * (ts.w * y.z + ts.z);
    }
    return make_float4(ox, oy, oz, 0.f);
}

// Skinning of the mesh vertices i0 + k stride (k < kLbsBatch, those below n):
// the streaming 128-bit loads of all of them are issued first (the mesh is
// read once per frame and bypasses L1), then each blends its frames (L2
// resident) and is written with a streaming 128-bit store.
constexpr int kLbsBatch = 2;
template <bool SHARED = false>
__device__ __forceinline__ void lbs_vertices(int i0, int stride, int n, int ns, const float4 *__restrict__ rest,
                                             const int4 *__restrict__ idx, const float4 *__restrict__ w,
                                             const float4 *__restrict__ frames, float4 *__restrict__ out, int *err)
{
    float4 p[kLbsBatch], ww[kLbsBatch];
    int4 id[kLbsBatch];
#pragma unroll
    for (int k = 0; k < kLbsBatch; ++k) {
        const int i = i0 + k * stride;
        if (i < n) {
            p[k] = __ldcs(rest + i);
            id[k] = __ldcs(idx + i);
            ww[k] = __ldcs(w + i);
        }
    }
#pragma unroll
    for (int k = 0; k < kLbsBatch; ++k) {
        const int i = i0 + k * stride;
        if (i < n) __stcs(out + i, lbs_blend<SHARED>(p[k], id[k], ww[k], ns, frames, err));
    }
}

}  // namespace viper
