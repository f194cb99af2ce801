// Trace kernels: one thread per ray, persistent warps pulling 8x4-pixel tiles, or parts of one, from a
// queue. Per ray: rounds of {pre-fill the k-buffer from the eviction list; traverse; blend the k-buffer
// in depth order with early termination} (Sec. III-A; Sec. IV-B, Listing 1). The first round, from the
// root, is traced for the whole warp: walked for the tile (tile_walk: checkpointed sphere-form traces
// without optional outputs) or as a packet (packet_round: the other forms, instrumented traces, every
// round of restart traversal). Later rounds go on from the checkpointed nodes, a ray a lane
// (trace_round). Rays of bundles that share nothing are walked one to a warp (k_trace_rays).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "grtx_internal.cuh"

// Scene arrays a trace reads (leaf order; see grtx_scene).
struct SceneRef {
    const float4 *nodes;
    const float4 *geom;
    const float4 *tris;
    const float *app;
    const uint32_t *gid;
    const float4 *tpl_nodes, *tpl_tris;   // icosphere forms: shared template BVH and triangles
    const float4 *raw;                    // [n_valid][3] raw parameters in leaf order (backward)
    const float4 *nodes4;                 // 4-wide nodes (8 float4 each), or NULL
    int app_stride, sh_degree, has_tree;
    uint32_t n_nodes, n_leaves, n_geom;   // internal nodes, leaf records, Gaussian records
    uint32_t n_nodes4;
};

// Leaf kinds of the trace kernels: one analytic unit sphere per Gaussian; one world-space
// proxy triangle per leaf (monolithic); one Gaussian instance whose leaf test traverses the
// shared icosphere template in unit-sphere space before the exact test.
// 3 and 4: sphere leaves under 4-wide nodes, with float or quantised child boxes
enum : int { FORM_SPHERE = 0, FORM_PROXY = 1, FORM_ICO = 2, FORM_SPHERE4 = 3, FORM_SPHERE4Q = 4 };

// A camera (rays generated in-kernel) or an explicit ray list.
struct CamRef {
    int cam_type, width, height, tiles_x;
    float3 pos, right, up, fwd;
    float tan_half, aspect, fish_f;
    float t_near, t_far;
    const float *ray_o, *ray_d, *ray_tn, *ray_tf;
};

struct TraceArgs {
    SceneRef sc;
    CamRef cam;
    unsigned n_items;            // queue items: 32 per warp tile (camera) or rays rounded up
    // parameters
    int traversal;               // GRTX_TRAVERSAL_*
    float T_min, alpha_max;
    float bg0, bg1, bg2;
    int ckpt_cap, evict_cap;
    int packet_stack;            // warp-stack entries a packet may use (1..kPacketStack)
    int window;                  // first round of a checkpointed ray: hits kept past the k-buffer (see Cut)
    float p_stop;                // product of (1 - alpha) below which a ray is known to terminate (see Cut)
    int id_shift;                // bits below the leaf slot in a list entry of windowed rays: kCodeBits or 0
    // per-slot workspace, interleaved [entry][slot]; the kernels address every list entry as
    // ck0[offset] with a 32-bit offset (ck1 = ck0 + ck1_off, ev = ck0 + ev_off; the host checks
    // that the whole workspace has fewer than 2^31 entries)
    uint2 *ck0, *ck1, *ev;
    uint32_t ck1_off, ev_off;
    int n_slots;
    int split;                   // k_trace: a warp takes 32 >> split rays at a time (see split_for)
    int middle;                  // tiles are handed out from the middle row outwards (see middle_out)
    int leave_at;                // work after which a bundle of several origins is left (see kWalkTrial)
    uint2 *left;                 // bundles left for k_trace_rays (counted in queue[4]), or NULL: the queue place, or
                                 // (batched views) the first item and the view
    int discard;                 // drop dead list lines from L2 after each tile (lists 256-byte aligned)
    unsigned *queue;
    unsigned long long *check;   // failed checks of the checked kernels (see in_bounds), or NULL
    // outputs
    float4 *rgbT;
    int32_t *n_blended;
    uint32_t *ids;
    int ids_cap;
    uint32_t *visits, *visits_n;   // visit log of sampled rays (see grtx_trace_outputs)
    int visits_cap, visits_stride, visits_rows;
    uint32_t *save_leaves;         // blend lists saved by a forward for its backward (grtx_saved)
    int32_t *save_n;
    int save_cap;
    grtx_stats *stats;
    // backward
    const float4 *fwd_rgbT, *dL_drgbT;
    const float *means, *log_scales, *quats, *logits;
    float *g_means, *g_log_scales, *g_quats, *g_logits, *g_sh;
    float4 *g_stage;             // [n_valid][3] per-leaf gradients of (mu, logit), log-scales, q
    int n_sh;
    int vec_sh;                  // gradients of SH (48 floats) may use float4 atomics
};

// One request of a serving step: its scene, camera, output, and which of its queue items
// this step covers (items [item_begin, item_begin + count) of the request map to step items
// [step_begin, step_begin + count)). Counts are multiples of 32. The kernel finds a tile's
// segment by a search over a separate array `begins` of the segments' step_begin values
// (ascending; entries past the last segment hold 0xffffffff, so that a launch's n_segs may be
// its table's capacity while the host appends segments).
// Records are 256-byte aligned so that a record the host appends while a launch runs shares
// no cache line with one the launch has already read.
struct __align__(256) ServeSeg {
    SceneRef sc;
    CamRef cam;
    float4 *out;
    unsigned item_begin, step_begin, count;
    unsigned split;              // batched ray lists: a 32-item tile of the queue stands for 32 >> split rays
};

// Controls of a serving launch (all NULL / 0 for a plain batched launch):
//   seg_done, seg_flag, seq: per-segment completion. The warp that finishes a segment's last
//     tile writes seq to seg_flag[segment] (pinned host memory mapped into the device).
//   avail: {items, closed}. The host appends segments while the launch runs: it writes their
//     records and begins entries, then raises the item count, and last, once it appends no
//     more, sets closed = 1. NULL: the launch's n_items is final. A warp claims its next tile
//     whether or not it is published yet and waits for it (sleeping between checks) until it
//     is published, the launch is closed, or linger_ns pass without any publication.
//   lost: [0] a count, then the first item of each tile a warp claimed and gave up on after
//     linger_ns; the host traces those again if it published them after all. lost_cap: the
//     launch's warps, since a warp stops after giving up.
//   exited: a count of warps that gave up, mirrored into exited_host (mapped host memory) so
//     that the host stops appending to a launch that has begun to wind down.
//   claimed_host: mapped host memory; every 16th claim, and every claim a warp has to wait
//     for, writes its end there, so that the host sees how much published work is left and
//     publishes more only when it runs low (the host chooses what runs next, instead of a long
//     queue fixing it).
static_assert(sizeof(ServeSeg) == 256, "a segment record fills one 256-byte slot");

struct ServeLive {
    unsigned *seg_done;
    unsigned *seg_flag;
    unsigned seq;
    const unsigned *avail;
    unsigned *lost;
    unsigned lost_cap;
    unsigned *exited;
    unsigned *exited_host;
    unsigned linger_ns;
    unsigned *claimed_host;
};

struct Counters {
    unsigned nodes, leaves, blended, rounds, ckpt, evictions, fallbacks, overflow;
    unsigned oob;      // fetch indices found outside their arrays (instrumented path only)
    uint32_t *vlog;    // the current ray's row of the visit log, or NULL (instrumented path only)
    unsigned vn, vcap;
};

// One node or leaf-record fetch of the current ray into its visit-log row (if it has one).
__device__ __forceinline__ void log_visit(Counters &c, uint32_t ref)
{
    if (c.vlog) {
        if (c.vn < c.vcap) c.vlog[c.vn] = ref;
        ++c.vn;
    }
}

// Self-check of the instrumented kernels (the ones that fill grtx_stats): before a node or
// leaf record is fetched its index is compared with the size of its array, and so is the
// Gaussian index a proxy triangle names. An index outside is counted (grtx_stats.bounds_errors)
// and not fetched; the traversal treats it as a miss. Every parity render runs these kernels,
// so every parity case is also a check that their traversal never leaves the scene's arrays. They
// take the first round as a packet: the walks, which the uninstrumented kernels take it by, have
// checked instantiations of their own (in_bounds, grtx_trace_self_check).
__device__ __forceinline__ bool ref_ok(const SceneRef &sc, uint32_t ref, Counters &c, bool count = true)
{
    bool ok = (ref & GRTX_LEAF) ? (ref & ~GRTX_LEAF) < sc.n_leaves : ref < sc.n_nodes;
    if (!ok && count) ++c.oob;
    return ok;
}

__device__ __forceinline__ bool ref4_ok(const SceneRef &sc, uint32_t ref, Counters &c, bool count = true)
{
    bool ok = (ref & GRTX_LEAF) ? (ref & ~GRTX_LEAF) < sc.n_leaves : ref < sc.n_nodes4;
    if (!ok && count) ++c.oob;
    return ok;
}

__device__ __forceinline__ bool gauss_ok(const SceneRef &sc, uint32_t gi, Counters &c)
{
    if (gi < sc.n_geom) return true;
    ++c.oob;
    return false;
}

// Check of the walks' checked instantiations (CHK): an index outside its array is counted in *a.check,
// and the caller leaves the access out.
template <bool CHK>
__device__ __forceinline__ bool in_bounds(const TraceArgs &a, uint32_t i, uint32_t n)
{
    if (!CHK || i < n) return true;
    atomicAdd(a.check, 1ull);
    return false;
}

#define GRTX_INF __int_as_float(0x7f800000)

// Start / finish the visit log of one ray (valid: the lane holds a ray with output index pix).
__device__ __forceinline__ void visits_begin(const TraceArgs &a, Counters &c, bool valid, int64_t pix)
{
    c.vlog = nullptr;
    c.vn = 0;
    if (a.visits && valid && pix % a.visits_stride == 0 && pix / a.visits_stride < a.visits_rows) {
        c.vlog = a.visits + (size_t)(pix / a.visits_stride) * a.visits_cap;
        c.vcap = (unsigned)a.visits_cap;
    }
}
__device__ __forceinline__ void visits_end(const TraceArgs &a, Counters &c, int64_t pix)
{
    if (c.vlog) a.visits_n[pix / a.visits_stride] = c.vn;
    c.vlog = nullptr;
}

// ------------------------------------------------------------------------------------------
// Rays
// ------------------------------------------------------------------------------------------
// Queue items: a warp's 32 items are an 8x4 pixel tile (tiles_x > 0: cameras, and ray lists
// laid out as an image of at least four rows, so that a warp's rays are neighbours), or 32
// consecutive rays of a list (tiles_x = 0). Output index pix = y * width + x either way.
__device__ __forceinline__ unsigned item_of_pixel(const CamRef &a, int64_t p)
{
    if (!a.tiles_x) return (unsigned)p;
    int x = (int)(p % a.width), y = (int)(p / a.width);
    return (unsigned)(((y / 4) * a.tiles_x + (x / 8)) * 32 + (y % 4) * 8 + (x % 8));
}

__device__ __forceinline__ bool make_ray(const CamRef &a, unsigned item, int64_t &pix, float3 &o, float3 &d,
                                         float &tn, float &tf)
{
    int px = 0, py = 0;
    if (a.tiles_x) {
        unsigned tile = item >> 5, l = item & 31u;
        px = (int)(tile % (unsigned)a.tiles_x) * 8 + (int)(l & 7u);
        py = (int)(tile / (unsigned)a.tiles_x) * 4 + (int)(l >> 3);
        if (px >= a.width || py >= a.height) return false;
        pix = (int64_t)py * a.width + px;
    } else {
        if ((int64_t)item >= (int64_t)a.width * a.height) return false;
        pix = item;
    }
    if (a.cam_type == GRTX_CAMERA_RAYS) {
        o = make_float3(a.ray_o[3 * pix], a.ray_o[3 * pix + 1], a.ray_o[3 * pix + 2]);
        d = make_float3(a.ray_d[3 * pix], a.ray_d[3 * pix + 1], a.ray_d[3 * pix + 2]);
        tn = a.ray_tn ? a.ray_tn[pix] : a.t_near;
        tf = a.ray_tf ? a.ray_tf[pix] : a.t_far;
        return true;
    }
    float dx, dy, dz;
    if (a.cam_type == GRTX_CAMERA_PINHOLE) {
        float u = (2.0f * (px + 0.5f) / a.width - 1.0f) * a.tan_half * a.aspect;
        float v = (1.0f - 2.0f * (py + 0.5f) / a.height) * a.tan_half;
        dx = a.fwd.x + u * a.right.x + v * a.up.x;
        dy = a.fwd.y + u * a.right.y + v * a.up.y;
        dz = a.fwd.z + u * a.right.z + v * a.up.z;
    } else {
        float ex = px + 0.5f - 0.5f * a.width, ey = 0.5f * a.height - (py + 0.5f);
        float r = sqrtf(ex * ex + ey * ey);
        float th = r / a.fish_f;
        float cp = r > 0.f ? ex / r : 1.f, sp = r > 0.f ? ey / r : 0.f;
        float st, ct;
        sincosf(th, &st, &ct);
        dx = st * cp * a.right.x + st * sp * a.up.x + ct * a.fwd.x;
        dy = st * cp * a.right.y + st * sp * a.up.y + ct * a.fwd.y;
        dz = st * cp * a.right.z + st * sp * a.up.z + ct * a.fwd.z;
    }
    float inv = rsqrtf(dx * dx + dy * dy + dz * dz);
    o = a.pos;
    d = make_float3(dx * inv, dy * inv, dz * inv);
    tn = a.t_near;
    tf = a.t_far;
    return true;
}

__device__ __forceinline__ float safe_rcp(float x)
{
    return fabsf(x) > 1e-30f ? 1.0f / x : copysignf(1e30f, x);
}

// ------------------------------------------------------------------------------------------
// k-buffer (Sec. III-A): the k nearest keys (t, leaf index) found so far, ascending. It lives in
// shared memory, entry j of thread x at [j * 128 + x], which keeps its 2k words out of the register
// file; t_max, the farthest kept depth once full, stays in a register. A key is one 64-bit number,
// the depth's bits mapped so that they order as the depths do, then the index: an insertion moves
// and compares whole keys (1M 1080p frame 3.51 -> 3.23 ms against separate depths and indices).
// Depths that compare equal have to have equal keys, so no depth may be -0 (see sphere_test).
// ------------------------------------------------------------------------------------------
constexpr int kBlock = 128;

__device__ __forceinline__ uint64_t make_key(float t, uint32_t i)
{
    const uint32_t b = __float_as_uint(t);
    return ((uint64_t)(b ^ ((uint32_t)((int)b >> 31) | 0x80000000u)) << 32) | i;
}
__device__ __forceinline__ float depth_of_key(uint64_t k)
{
    const uint32_t b = (uint32_t)(k >> 32);
    return __uint_as_float(b ^ (~(uint32_t)((int)b >> 31) | 0x80000000u));
}

template <int K>
struct KBuf {
    uint64_t *k;
    int n;
    float tmax;
    __device__ __forceinline__ void clear()
    {
        n = 0;
        tmax = GRTX_INF;
    }
    __device__ __forceinline__ float T(int j) const { return depth_of_key(k[j * kBlock]); }
    __device__ __forceinline__ uint32_t I(int j) const { return (uint32_t)k[j * kBlock]; }
    __device__ __forceinline__ bool contains(float ct, uint32_t ci) const
    {
        const uint64_t key = make_key(ct, ci);
        for (int j = 0; j < n; ++j)
            if (k[j * kBlock] == key) return true;
        return false;
    }
    // Insert (ct, ci) in key order. When the buffer was already full the larger of {new key,
    // farthest kept key} is rejected: it is returned in (ct, ci) and the result is true.
    __device__ __forceinline__ bool insert(float &ct, uint32_t &ci)
    {
        const uint64_t key = make_key(ct, ci);
        int pos;
        bool rejected = false;
        if (n == K) {
            const uint64_t last = k[(K - 1) * kBlock];
            if (key >= last) return true;
            ct = depth_of_key(last);
            ci = (uint32_t)last;
            rejected = true;
            pos = K - 1;
        } else {
            pos = n++;
        }
        while (pos > 0) {
            const uint64_t before = k[(pos - 1) * kBlock];
            if (before <= key) break;
            k[pos * kBlock] = before;
            --pos;
        }
        k[pos * kBlock] = key;
        if (n == K) tmax = depth_of_key(k[(K - 1) * kBlock]);
        return rejected;
    }
};

// How far a checkpointed ray still has to look. P is the product of (1 - alpha) over every hit
// it has collected (blended, in the k-buffer or on the eviction list; each hit is collected
// once) and far their farthest depth. Once P is below p_stop, just under T_min, the ray ends at
// or before `far`: hits and nodes beyond it can never be blended, and are dropped, not
// checkpointed. (p_stop = 0.98 T_min: P and the blended T round the same factors in different
// orders, each product of n factors within n 2^-23 of the exact one, and a ray's lists hold
// fewer than 2^17 hits.)
constexpr int kCodeBits = 8;

// -log2(q) of a hit's q = 1 - alpha in 8 bits, rounded down: exponents 2^-20 to 2^11 with 3 bits of
// mantissa, 0 for anything below. Scenes of fewer than 2^24 leaf slots keep it below the slot in a
// ray's list entries (slot << 8 | code, which orders as the slot does; see squeeze).
__device__ __forceinline__ uint32_t opacity_code(float q)
{
    const int c = (int)((__float_as_uint(__log2f(q)) & 0x7fffffffu) >> 20) - (107 << 3);
    return (uint32_t)min(max(c, 0), 255);
}
__device__ __forceinline__ float opacity_of_code(uint32_t c)
{
    return c ? __uint_as_float((c + (107u << 3)) << 20) : 0.f;
}

struct Cut {
    float P, far;
    __device__ __forceinline__ void clear()
    {
        P = 1.0f;
        far = 0.0f;
    }
    __device__ __forceinline__ float top(const TraceArgs &a) const { return P < a.p_stop ? far : GRTX_INF; }
    // Counts a hit of Gaussian record g (leaf slot gi) and returns the slot as the lists hold it.
    __device__ __forceinline__ uint32_t add(const TraceArgs &a, const float4 *__restrict__ g, uint32_t gi, float t, float D2)
    {
        const float4 r3 = __ldg(g + 3);
        return take(a, 1.0f - fminf(r3.x * exp2f(r3.y * D2), a.alpha_max), gi, t);
    }
    __device__ __forceinline__ uint32_t take(const TraceArgs &a, float q, uint32_t gi, float t)      // q = 1 - alpha
    {
        P *= q;
        far = fmaxf(far, t);
        return a.id_shift ? gi << kCodeBits | opacity_code(q) : gi;
    }
};

__device__ __forceinline__ bool key_after(float t, uint32_t i, float Lt, uint32_t Li)
{
    return t > Lt || (t == Lt && i > Li);
}

// Two consecutive float4 in one 256-bit load (p 32-byte aligned: nodes, records and rows of 48
// coefficients are). Where each lane gathers a record of its own, the L1 pipe (78 % busy on the 1M
// 1080p frame) takes a pass for every line that a load touches, so half the loads are half the passes.
// The walk's nodes, the filter's and the exact test's records and the blend's: frame 3.25 -> 3.19 ms.
// The colour's rows only in the backward (training step 2.60 -> 2.56 ms): the forward kernel has no
// eight registers to spare for them (frame +0.5 %).
__device__ __forceinline__ void ldg2(const float4 *p, float4 &a, float4 &b)
{
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}
// Closest approach of the ray to the centre of a Gaussian in its unit-sphere space (Sec. IV-A):
// with the record rows (A_j | mu_j), o_l = A (o - mu), d_l = A d, t = -(o_l.d_l)/(d_l.d_l) and
// D2 = |o_l + t d_l|^2. t is the max-response depth of Sec. III-A Eq. t-max-resp, and D2 <= 1
// iff alpha >= alpha_min. Stage 1 runs for every leaf and only filters: in FP32 its absolute
// error in D2 grows like |o_l| (the ray origin measured in Gaussian widths), so the threshold
// is widened to 1 + 1e-5 + 4e-6 |o_l|, tested in squared form (no square root). Its t only
// seeds stage 2, whose Newton step lands on the minimiser from any nearby start, so the
// quotient is the fast approximate one.
__device__ __forceinline__ bool sphere_candidate(float4 r0, float4 r1, float4 r2, float3 o, float3 d, float &t,
                                                 float &aa)
{
    float vx = o.x - r0.w, vy = o.y - r1.w, vz = o.z - r2.w;
    float olx = fmaf(r0.x, vx, fmaf(r0.y, vy, r0.z * vz));
    float oly = fmaf(r1.x, vx, fmaf(r1.y, vy, r1.z * vz));
    float olz = fmaf(r2.x, vx, fmaf(r2.y, vy, r2.z * vz));
    float dlx = fmaf(r0.x, d.x, fmaf(r0.y, d.y, r0.z * d.z));
    float dly = fmaf(r1.x, d.x, fmaf(r1.y, d.y, r1.z * d.z));
    float dlz = fmaf(r2.x, d.x, fmaf(r2.y, d.y, r2.z * d.z));
    aa = fmaf(dlx, dlx, fmaf(dly, dly, dlz * dlz));
    float bb = fmaf(olx, dlx, fmaf(oly, dly, olz * dlz));
    t = __fdividef(-bb, aa);
    float px = fmaf(t, dlx, olx), py = fmaf(t, dly, oly), pz = fmaf(t, dlz, olz);
    float D2 = fmaf(px, px, fmaf(py, py, pz * pz));
    float oo = fmaf(olx, olx, fmaf(oly, oly, olz * olz));
    float ex = D2 - (1.0f + 1e-5f);
    return ex <= 0.0f || ex * ex <= 1.6e-11f * oo;    // ex <= 4e-6 sqrt(oo)
}
__device__ __forceinline__ bool sphere_candidate(float4 r0, float4 r1, float4 r2, float3 o, float3 d, float &t)
{
    float aa;
    return sphere_candidate(r0, r1, r2, o, d, t, aa);
}

// Whether the depth t of sphere_candidate may stand for an exact depth in (lo, hi]. Its error is the
// rounding of o - mu taken through A, a few ulp of |t| and of the half chord 1 / |d_l| times the
// Gaussian's aspect ratio, and of A d once the ratio comes near 2^23: 1e-5, 5e-4 and 0.036 of both at
// ratios of 10^3, 10^5 and 3 10^6 (largest of 4 10^5 rays in a disc's plane, against 64 bits). An eighth
// of both is taken; beyond that sphere_candidate itself loses hits.
__device__ __forceinline__ bool in_range(float t, float aa, float lo, float hi)
{
    const float m = 0.125f * (fabsf(t) + rsqrtf(aa));
    return !(t + m < lo) && !(t - m > hi);
}

// Error-free a + b = s + e (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float a, float b, float &e)
{
    float s = __fadd_rn(a, b);
    float bv = __fsub_rn(s, a);
    float av = __fsub_rn(s, bv);
    e = __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
    return s;
}

// Stage 2 for candidates: the world offset w = o + t d - mu is formed as an unevaluated sum of
// two floats (two-sum for o - mu, an FMA for the rounding error of t d), mapped to unit-sphere
// space, and t is moved to the exact minimiser along the line by one Newton step. D2 is then
// accurate to a few ulp of 1 whatever the distance from the ray origin. w receives the world
// offset of the closest point from the mean.
__device__ __forceinline__ void sphere_refine(float4 r0, float4 r1, float4 r2, float3 o, float3 d, float &t, float &D2,
                                              float w[3])
{
    const float oc[3] = {o.x, o.y, o.z}, dc[3] = {d.x, d.y, d.z}, mu[3] = {r0.w, r1.w, r2.w};
    float wh[3], wl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float vl, e1;
        float vh = two_sum(oc[c], -mu[c], vl);
        float ph = __fmul_rn(t, dc[c]);
        float pl = fmaf(t, dc[c], -ph);
        wh[c] = two_sum(vh, ph, e1);
        wl[c] = e1 + vl + pl;
    }
    const float4 R[3] = {r0, r1, r2};
    float p[3], dl[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        float lo = fmaf(R[j].x, wl[0], fmaf(R[j].y, wl[1], R[j].z * wl[2]));
        p[j] = fmaf(R[j].x, wh[0], fmaf(R[j].y, wh[1], fmaf(R[j].z, wh[2], lo)));
        dl[j] = fmaf(R[j].x, d.x, fmaf(R[j].y, d.y, R[j].z * d.z));
    }
    // the step only corrects t, so the fast quotient's few-ulp relative error in it stays far
    // below one ulp of t
    float delta = __fdividef(fmaf(p[0], dl[0], fmaf(p[1], dl[1], p[2] * dl[2])),
                             fmaf(dl[0], dl[0], fmaf(dl[1], dl[1], dl[2] * dl[2])));
    t -= delta;
#pragma unroll
    for (int j = 0; j < 3; ++j) p[j] = fmaf(-delta, dl[j], p[j]);
    D2 = fmaf(p[0], p[0], fmaf(p[1], p[1], p[2] * p[2]));
#pragma unroll
    for (int c = 0; c < 3; ++c) w[c] = fmaf(-delta, dc[c], wh[c] + wl[c]);
}

// Full test of one Gaussian record: returns true for a hit candidate and then (t, D2, w). A depth of -0
// becomes +0: a ray that starts at the mean of several Gaussians has zeros of either sign among its
// depths, and a round goes on behind the last key's depth and index (key_after), which compares them as
// equal. (The tile walk takes no ray with t_near < 0, hence has no such depth.)
__device__ __forceinline__ bool sphere_test(const float4 *__restrict__ g, float3 o, float3 d, float &t, float &D2,
                                            float w[3])
{
    float4 r0 = __ldg(g), r1 = __ldg(g + 1), r2 = __ldg(g + 2);
    if (!sphere_candidate(r0, r1, r2, o, d, t)) return false;
    sphere_refine(r0, r1, r2, o, d, t, D2, w);
    t = __fadd_rn(t, 0.0f);
    return true;
}

// Real spherical harmonics up to degree 3 (no Condon-Shortley phase), index l*l + l + m,
// times the coefficients: c = max(0, sum_k Y_k(dir) f_k + 0.5); raw receives the sum + 0.5.
// The record holds the coefficients as (k, channel) pairs padded to a multiple of 4 floats
// and is read with float4 loads.
template <bool WIDE = false>
__device__ __forceinline__ void sh_color(const float *__restrict__ f, int deg, int stride, float3 n, float c[3],
                                         float raw[3], float Y[16])
{
    float x = n.x, y = n.y, z = n.z;
#pragma unroll
    for (int k = 0; k < 16; ++k) Y[k] = 0.f;
    Y[0] = 0.28209479177387814f;
    if (deg >= 1) {
        Y[1] = 0.4886025119029199f * y;
        Y[2] = 0.4886025119029199f * z;
        Y[3] = 0.4886025119029199f * x;
    }
    if (deg >= 2) {
        Y[4] = 1.0925484305920792f * x * y;
        Y[5] = 1.0925484305920792f * y * z;
        Y[6] = 0.31539156525252005f * (3.f * z * z - 1.f);
        Y[7] = 1.0925484305920792f * x * z;
        Y[8] = 0.5462742152960396f * (x * x - y * y);
    }
    if (deg >= 3) {
        Y[9] = 0.5900435899266435f * y * (3.f * x * x - y * y);
        Y[10] = 2.890611442640554f * x * y * z;
        Y[11] = 0.4570457994644658f * y * (5.f * z * z - 1.f);
        Y[12] = 0.3731763325901154f * z * (5.f * z * z - 3.f);
        Y[13] = 0.4570457994644658f * x * (5.f * z * z - 1.f);
        Y[14] = 1.445305721320277f * z * (x * x - y * y);
        Y[15] = 0.5900435899266435f * x * (x * x - 3.f * y * y);
    }
    float acc[3] = {0.5f, 0.5f, 0.5f};
    const int n_vec = stride >> 2;
    const float4 *f4 = reinterpret_cast<const float4 *>(f);
    if (WIDE && n_vec == 12) {
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            float4 u, v;
            ldg2(f4 + 2 * j, u, v);
            const float qq[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = 8 * j + e;                    // flat index = 3 k + channel
                acc[i % 3] = fmaf(Y[i / 3], qq[e], acc[i % 3]);
            }
        }
    } else
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        if (j < n_vec) {
            float4 q = __ldg(f4 + j);
            const float qq[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = 4 * j + e;                // flat index = 3 k + channel
                if (i < 48) acc[i % 3] = fmaf(Y[i / 3], qq[e], acc[i % 3]);
            }
        }
    }
    raw[0] = acc[0]; raw[1] = acc[1]; raw[2] = acc[2];
    c[0] = fmaxf(acc[0], 0.f); c[1] = fmaxf(acc[1], 0.f); c[2] = fmaxf(acc[2], 0.f);
}

// Slab test of one child box against the ray over [tn, tf]: entry / exit distances, each
// plane distance as one FMA, l * inv - o * inv. Its rounding error is an ulp of the origin's
// plane distance, far inside the margin between a box's entry and the depth of any Gaussian hit
// in it, except for grazing hits at alpha_min; an axis-parallel ray (inv = 1e30) lying exactly
// in a face plane may lose that box, which it could only touch tangentially.
__device__ __forceinline__ void slab(float lx, float ly, float lz, float hx, float hy, float hz, float3 o, float3 inv,
                                     float tn, float tf, float &t0, float &t1)
{
    const float px = -o.x * inv.x, py = -o.y * inv.y, pz = -o.z * inv.z;
    float ax = fmaf(lx, inv.x, px), bx = fmaf(hx, inv.x, px);
    float ay = fmaf(ly, inv.y, py), by = fmaf(hy, inv.y, py);
    float az = fmaf(lz, inv.z, pz), bz = fmaf(hz, inv.z, pz);
    t0 = fmaxf(fmaxf(fminf(ax, bx), fminf(ay, by)), fmaxf(fminf(az, bz), tn));
    t1 = fminf(fminf(fmaxf(ax, bx), fmaxf(ay, by)), fminf(fmaxf(az, bz), tf));
}

// Ray / triangle (Moller-Trumbore) with a small barycentric tolerance so that shared edges
// of the proxy never leak; returns the hit distance or +inf.
__device__ __forceinline__ float tri_hit(float4 v0, float4 v1, float4 v2, float3 o, float3 d)
{
    float e1x = v1.x - v0.x, e1y = v1.y - v0.y, e1z = v1.z - v0.z;
    float e2x = v2.x - v0.x, e2y = v2.y - v0.y, e2z = v2.z - v0.z;
    float px = d.y * e2z - d.z * e2y, py = d.z * e2x - d.x * e2z, pz = d.x * e2y - d.y * e2x;
    float det = e1x * px + e1y * py + e1z * pz;
    if (fabsf(det) < 1e-30f) return GRTX_INF;
    float id = 1.0f / det;
    float sx = o.x - v0.x, sy = o.y - v0.y, sz = o.z - v0.z;
    float u = (sx * px + sy * py + sz * pz) * id;
    const float eps = 1e-5f;
    if (u < -eps || u > 1.f + eps) return GRTX_INF;
    float qx = sy * e1z - sz * e1y, qy = sz * e1x - sx * e1z, qz = sx * e1y - sy * e1x;
    float v = (d.x * qx + d.y * qy + d.z * qz) * id;
    if (v < -eps || u + v > 1.f + eps) return GRTX_INF;
    return (e2x * qx + e2y * qy + e2z * qz) * id;
}

// Leaf test of the instanced-icosphere forms (Sec. IV-A, second option): the ray in Gaussian
// gi's unit-sphere space (o_l = A (o - mu), d_l = A d, so t is the world t) traverses the
// shared template BVH; true at the first template triangle hit beyond t_near. The local ray
// is scaled by 1 / (1 + 1e-5 + 4e-6 |o_l|), which inflates the template against the FP32
// error of o_l without changing t, so that no exact hit is lost.
template <bool INSTR>
__device__ __forceinline__ bool template_touch(const SceneRef &sc, uint32_t gi, float3 o, float3 d, float tn,
                                               Counters &cnt)
{
    const float4 *g = sc.geom + 4 * (size_t)gi;
    float4 r0 = __ldg(g), r1 = __ldg(g + 1), r2 = __ldg(g + 2);
    float rx = o.x - r0.w, ry = o.y - r1.w, rz = o.z - r2.w;
    float3 ol = make_float3(r0.x * rx + r0.y * ry + r0.z * rz, r1.x * rx + r1.y * ry + r1.z * rz,
                            r2.x * rx + r2.y * ry + r2.z * rz);
    float sc_l = 1.0f / (1.0f + 1e-5f + 4e-6f * sqrtf(ol.x * ol.x + ol.y * ol.y + ol.z * ol.z));
    ol = make_float3(ol.x * sc_l, ol.y * sc_l, ol.z * sc_l);
    float3 dl = make_float3((r0.x * d.x + r0.y * d.y + r0.z * d.z) * sc_l, (r1.x * d.x + r1.y * d.y + r1.z * d.z) * sc_l,
                            (r2.x * d.x + r2.y * d.y + r2.z * d.z) * sc_l);
    float3 inv = make_float3(safe_rcp(dl.x), safe_rcp(dl.y), safe_rcp(dl.z));
    uint32_t stack[16];
    int sp = 0;
    uint32_t ref = 0u;
    for (;;) {
        if (ref & GRTX_LEAF) {
            if (INSTR) cnt.leaves++;
            const float4 *tr = sc.tpl_tris + 3 * (size_t)(ref & ~GRTX_LEAF);
            if (tri_hit(__ldg(tr), __ldg(tr + 1), __ldg(tr + 2), ol, dl) > tn) return true;
        } else {
            if (INSTR) cnt.nodes++;
            const float4 *nd = sc.tpl_nodes + 4 * (size_t)ref;
            float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
            float e0, x0, e1, x1;
            slab(n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, ol, inv, tn, GRTX_INF, e0, x0);
            slab(n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, ol, inv, tn, GRTX_INF, e1, x1);
            bool h0 = e0 <= x0, h1 = e1 <= x1;
            uint32_t c0 = __float_as_uint(n3.x), c1 = __float_as_uint(n3.y);
            if (h0 && h1) {
                bool near0 = e0 <= e1;
                ref = near0 ? c0 : c1;
                if (sp < 16) stack[sp++] = near0 ? c1 : c0;
                continue;
            }
            if (h0 || h1) {
                ref = h0 ? c0 : c1;
                continue;
            }
        }
        if (sp == 0) return false;
        ref = stack[--sp];
    }
}

// ------------------------------------------------------------------------------------------
// 4-wide nodes (FORM_SPHERE4; see grtx_params.bvh_width). A node holds its four children's
// boxes as per-axis rows; empty children have empty boxes (lo = +inf, hi = -inf) and ref
// GRTX_NONE. The rounds are those of the binary traversal: a child whose entry exceeds t_max
// is checkpointed, the others are visited, nearest first.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float pick4(const float v[4], int i)
{
    return i == 0 ? v[0] : (i == 1 ? v[1] : (i == 2 ? v[2] : v[3]));
}
__device__ __forceinline__ uint32_t pick4(const uint32_t v[4], int i)
{
    return i == 0 ? v[0] : (i == 1 ? v[1] : (i == 2 ? v[2] : v[3]));
}

// Float4 words of one 4-wide node: 8 with float child boxes, 4 with quantised ones.
template <bool Q>
__device__ __forceinline__ const float4 *node4(const SceneRef &sc, uint32_t ref)
{
    return sc.nodes4 + (Q ? 4 : 8) * (size_t)ref;
}

// Decoded quantised box coordinate: the node's corner plus q steps (one FMA, exactly as the
// build checked it). eb: the step's biased exponent.
__device__ __forceinline__ float dq(uint32_t q, uint32_t eb, float o)
{
    return fmaf(__uint2float_rn(q), __uint_as_float(eb << 23), o);
}

// Entry and exit of the ray in each child box of a 4-wide node (e > x: missed).
template <bool Q>
__device__ __forceinline__ void slab4(const float4 *__restrict__ nd, float3 o, float3 inv, float tn, float tf, float e[4],
                                      float x[4], uint32_t c[4])
{
    if (Q) {
        const float4 h = __ldg(nd);
        const uint4 qa = __ldg(reinterpret_cast<const uint4 *>(nd + 1));
        const uint4 qb = __ldg(reinterpret_cast<const uint4 *>(nd + 2));
        const uint4 qc = __ldg(reinterpret_cast<const uint4 *>(nd + 3));
        const uint32_t eb = __float_as_uint(h.w);
        const uint32_t ex = eb & 0xffu, ey = (eb >> 8) & 0xffu, ez = (eb >> 16) & 0xffu;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int sh = 8 * j;
            slab(dq((qa.x >> sh) & 0xffu, ex, h.x), dq((qa.y >> sh) & 0xffu, ey, h.y), dq((qa.z >> sh) & 0xffu, ez, h.z),
                 dq((qa.w >> sh) & 0xffu, ex, h.x), dq((qb.x >> sh) & 0xffu, ey, h.y), dq((qb.y >> sh) & 0xffu, ez, h.z),
                 o, inv, tn, tf, e[j], x[j]);
        }
        c[0] = qb.z;
        c[1] = qb.w;
        c[2] = qc.x;
        c[3] = qc.y;
        return;
    }
    const float4 lx = __ldg(nd), ly = __ldg(nd + 1), lz = __ldg(nd + 2);
    const float4 hx = __ldg(nd + 3), hy = __ldg(nd + 4), hz = __ldg(nd + 5);
    const float4 rf = __ldg(nd + 6);
    slab(lx.x, ly.x, lz.x, hx.x, hy.x, hz.x, o, inv, tn, tf, e[0], x[0]);
    slab(lx.y, ly.y, lz.y, hx.y, hy.y, hz.y, o, inv, tn, tf, e[1], x[1]);
    slab(lx.z, ly.z, lz.z, hx.z, hy.z, hz.z, o, inv, tn, tf, e[2], x[2]);
    slab(lx.w, ly.w, lz.w, hx.w, hy.w, hz.w, o, inv, tn, tf, e[3], x[3]);
    c[0] = __float_as_uint(rf.x);
    c[1] = __float_as_uint(rf.y);
    c[2] = __float_as_uint(rf.z);
    c[3] = __float_as_uint(rf.w);
}

// Order (key, ord) pairs ascending by key: a 5-comparator network over 4 entries.
__device__ __forceinline__ void sort4(float k[4], int ord[4])
{
#define GRTX_CSWAP(i, j)                                                              \
    if (k[j] < k[i]) {                                                                \
        float tk = k[i]; k[i] = k[j]; k[j] = tk;                                      \
        int to = ord[i]; ord[i] = ord[j]; ord[j] = to;                                \
    }
    GRTX_CSWAP(0, 1) GRTX_CSWAP(2, 3) GRTX_CSWAP(0, 2) GRTX_CSWAP(1, 3) GRTX_CSWAP(1, 2)
#undef GRTX_CSWAP
}

// The sphere-leaf test of one leaf slot inside a round (shared by the 4-wide traversals):
// a hit with key in (L, t_max] enters the k-buffer; a hit the full buffer rejects goes to the
// eviction list when checkpointing. Returns false when the eviction list would overflow.
template <int K, bool INSTR>
__device__ __forceinline__ bool leaf4(const TraceArgs &a, const SceneRef &sc, uint32_t ref, float3 o, float3 d, float tn,
                                      float tf, float Lt, uint32_t Li, bool ckpt, uint32_t ev, int &n_ev, KBuf<K> &kb,
                                      float &tmax, Counters &cnt)
{
    const uint32_t gi = ref & ~GRTX_LEAF;
    if (INSTR) {
        cnt.leaves++;
        log_visit(cnt, ref);
    }
    float t, D2, w[3];
    if (sphere_test(sc.geom + 4 * (size_t)gi, o, d, t, D2, w) && D2 <= 1.0f && t > tn && t <= tf &&
        key_after(t, gi, Lt, Li)) {
        float ct = t;
        uint32_t ci = gi;
        if (kb.insert(ct, ci) && ckpt) {
            if (n_ev >= a.evict_cap) return false;
            a.ck0[ev + (uint32_t)n_ev * (uint32_t)a.n_slots] = make_uint2(__float_as_uint(ct), ci);
            ++n_ev;
            if (INSTR) cnt.evictions++;
        }
        tmax = kb.tmax;
    }
    return true;
}

// Entry distance of the ray into child `slot` of 4-wide node `parent`.
template <bool Q>
__device__ __forceinline__ float child_entry4(const SceneRef &sc, uint32_t parent, uint32_t slot, float3 o, float3 inv,
                                              float tn, float tf)
{
    float te, x;
    if (Q) {
        const float4 *nd = node4<true>(sc, parent);
        const float4 h = __ldg(nd);
        const uint4 qa = __ldg(reinterpret_cast<const uint4 *>(nd + 1));
        const uint4 qb = __ldg(reinterpret_cast<const uint4 *>(nd + 2));
        const uint32_t eb = __float_as_uint(h.w), sh = 8 * slot;
        const uint32_t ex = eb & 0xffu, ey = (eb >> 8) & 0xffu, ez = (eb >> 16) & 0xffu;
        slab(dq((qa.x >> sh) & 0xffu, ex, h.x), dq((qa.y >> sh) & 0xffu, ey, h.y), dq((qa.z >> sh) & 0xffu, ez, h.z),
             dq((qa.w >> sh) & 0xffu, ex, h.x), dq((qb.x >> sh) & 0xffu, ey, h.y), dq((qb.y >> sh) & 0xffu, ez, h.z), o,
             inv, tn, tf, te, x);
    } else {
        const float *pn = reinterpret_cast<const float *>(node4<false>(sc, parent));
        slab(__ldg(pn + slot), __ldg(pn + 4 + slot), __ldg(pn + 8 + slot), __ldg(pn + 12 + slot), __ldg(pn + 16 + slot),
             __ldg(pn + 20 + slot), o, inv, tn, tf, te, x);
    }
    return te;
}

// One round of one ray over 4-wide nodes (the per-ray rounds; see trace_round).
template <int K, bool INSTR, bool Q>
__device__ __forceinline__ bool trace_round4(const TraceArgs &a, const SceneRef &sc, float3 o, float3 d, float3 inv,
                                             float tn, float tf, float Lt, uint32_t Li, bool ckpt, bool from_root,
                                             uint32_t src, int n_src, uint32_t dst, int &n_dst, uint32_t ev,
                                             int &n_ev, KBuf<K> &kb, Counters &cnt)
{
    const uint32_t S = (uint32_t)a.n_slots;
    uint2 *__restrict__ const L = a.ck0;
    uint32_t stack[GRTX_STACK4];               // node refs; a popped entry is visited (see trace_round)
    int sp = 0, si = 0;
    float tmax = kb.tmax;
    uint32_t ref;
    float te;
    n_dst = 0;
    if (from_root) {
        n_src = 0;
        ref = 0u;
        te = tn;
    } else {
        if (n_src == 0) return true;
        uint2 v = L[src];
        ref = v.x;
        te = __uint_as_float(v.y);
        si = 1;
    }
    for (;;) {
        if (te > tmax) {
            if (ckpt) {
                if (n_dst >= a.ckpt_cap) return false;
                L[dst + (uint32_t)n_dst * S] = make_uint2(ref, __float_as_uint(te));
                ++n_dst;
                if (INSTR) cnt.ckpt++;
            }
        } else if (INSTR && !ref4_ok(sc, ref, cnt)) {
        } else if (ref & GRTX_LEAF) {
            if (!leaf4<K, INSTR>(a, sc, ref, o, d, tn, tf, Lt, Li, ckpt, ev, n_ev, kb, tmax, cnt)) return false;
        } else {
            if (INSTR) {
                cnt.nodes++;
                log_visit(cnt, ref);
            }
            float e[4], x[4];
            uint32_t c[4];
            slab4<Q>(node4<Q>(sc, ref), o, inv, tn, tf, e, x, c);
            int ord[4] = {0, 1, 2, 3};
            int nh = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool h = e[j] <= x[j] && !(x[j] < Lt) && c[j] != GRTX_NONE;
                nh += h;
                if (!h) e[j] = GRTX_INF;           // misses sort last
            }
            if (nh > 0) {
                sort4(e, ord);
#pragma unroll
                for (int j = 3; j >= 1; --j) {    // farthest first onto the stack, so the nearest pops first
                    if (j < nh) {
                        const uint32_t cj = pick4(c, ord[j]);
                        if (e[j] > tmax) {
                            if (ckpt) {
                                if (n_dst >= a.ckpt_cap) return false;
                                L[dst + (uint32_t)n_dst * S] = make_uint2(cj, __float_as_uint(e[j]));
                                ++n_dst;
                                if (INSTR) cnt.ckpt++;
                            }
                        } else if (sp < GRTX_STACK4) {
                            stack[sp++] = cj;
                        } else if (INSTR) {
                            cnt.overflow++;
                        }
                    }
                }
                ref = pick4(c, ord[0]);
                te = e[0];
                continue;
            }
        }
        if (sp > 0) {
            ref = stack[--sp];
            te = -GRTX_INF;
        } else if (si < n_src) {
            uint2 v = L[src + (uint32_t)si * S];
            ++si;
            ref = v.x;
            te = __uint_as_float(v.y);
        } else {
            break;
        }
    }
    return true;
}

// A round of a warp's rays from the root as one packet over 4-wide nodes (see packet_round).
// At a node every lane tests the four children; the warp continues into the child its lowest
// active lane enters first and keeps the others, with the lanes that want them, on the warp's
// stack (entries: child, parent << 2 | child slot, lane mask); a popped child's entry
// distance is recomputed per lane from its box in the parent.
template <int K, bool INSTR, bool Q>
__device__ __forceinline__ bool packet_round4(const TraceArgs &a, const SceneRef &sc, bool valid, uint4 *pst, float3 o,
                                              float3 d, float3 inv, float tn, float tf, float Lt, uint32_t Li,
                                              bool ckpt, uint32_t dst, int &n_dst, uint32_t ev, int &n_ev, KBuf<K> &kb,
                                              Counters &cnt, bool &lane_ok)
{
    const unsigned full = 0xffffffffu;
    const uint32_t S = (uint32_t)a.n_slots;
    uint2 *__restrict__ const L = a.ck0;
    const int lane = threadIdx.x & 31;
    float tmax = kb.tmax;
    n_dst = 0;
    n_ev = 0;
    lane_ok = true;
    if (!sc.has_tree) return true;
    int sp = 0;
    uint32_t ref = 0u, parent = GRTX_NONE, slot = 0u;
    unsigned m = __ballot_sync(full, valid);
    float te = tn;
    bool have_te = true;
    for (;;) {
        const bool in = (m >> lane) & 1u;
        if (!have_te && in) te = child_entry4<Q>(sc, parent, slot, o, inv, tn, tf);   // a popped child
        const bool go = in && lane_ok && !(te > tmax);
        if (in && lane_ok && te > tmax && ckpt) {
            if (n_dst >= a.ckpt_cap) {
                lane_ok = false;
            } else {
                L[dst + (uint32_t)n_dst * S] = make_uint2(ref, __float_as_uint(te));
                ++n_dst;
                if (INSTR) cnt.ckpt++;
            }
        }
        m = __ballot_sync(full, go);
        bool pop = true;
        if (m && (!INSTR || ref4_ok(sc, ref, cnt, go))) {   // ref is the warp's: all lanes agree
            if (ref & GRTX_LEAF) {
                if (go && !leaf4<K, INSTR>(a, sc, ref, o, d, tn, tf, Lt, Li, ckpt, ev, n_ev, kb, tmax, cnt))
                    lane_ok = false;
            } else {
                float e[4], x[4];
                uint32_t c[4];
                slab4<Q>(node4<Q>(sc, ref), o, inv, tn, tf, e, x, c);
                bool h[4];
                unsigned mh[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    h[j] = go && e[j] <= x[j] && !(x[j] < Lt) && c[j] != GRTX_NONE;
                    mh[j] = __ballot_sync(full, h[j]);
                }
                if (INSTR && go) {
                    cnt.nodes++;
                    log_visit(cnt, ref);
                }
                // order the wanted children by the lowest active lane's entry distances (children
                // it misses after those it enters, in child order; children nobody wants last)
                const int leader = __ffs(m) - 1;
                float k2[4];
                int rk[4], ord[4] = {0, 1, 2, 3};
                int nc = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float kl = __shfl_sync(full, h[j] ? e[j] : GRTX_INF, leader);
                    rk[j] = mh[j] == 0u ? 2 : (kl < GRTX_INF ? 0 : 1);
                    k2[j] = kl;
                    nc += mh[j] != 0u;
                }
                if (nc > 0) {
#define GRTX_CSWAP4(i, j)                                                                                 \
    if (rk[j] < rk[i] || (rk[j] == rk[i] && rk[i] == 0 && k2[j] < k2[i])) {                            \
        int tr = rk[i]; rk[i] = rk[j]; rk[j] = tr;                                                        \
        float tk = k2[i]; k2[i] = k2[j]; k2[j] = tk;                                                      \
        int to = ord[i]; ord[i] = ord[j]; ord[j] = to;                                                    \
    }
                    GRTX_CSWAP4(0, 1) GRTX_CSWAP4(2, 3) GRTX_CSWAP4(0, 2) GRTX_CSWAP4(1, 3) GRTX_CSWAP4(1, 2)
#undef GRTX_CSWAP4
                    if (sp + nc - 1 > a.packet_stack) {       // too deep for the warp's stack
                        lane_ok = false;
                        return false;
                    }
                    if (lane == 0) {
#pragma unroll
                        for (int j = 3; j >= 1; --j) {        // farthest first
                            if (j < nc) {
                                const int oj = ord[j];
                                pst[sp + (nc - 1 - j)] = make_uint4(pick4(c, oj), (ref << 2) | (uint32_t)oj,
                                                                    oj == 0 ? mh[0] : (oj == 1 ? mh[1] : (oj == 2 ? mh[2] : mh[3])), 0u);
                            }
                        }
                    }
                    sp += nc - 1;
                    __syncwarp(full);
                    const int f = ord[0];
                    parent = ref;
                    slot = (uint32_t)f;
                    m = f == 0 ? mh[0] : (f == 1 ? mh[1] : (f == 2 ? mh[2] : mh[3]));
                    te = pick4(e, f);
                    ref = pick4(c, f);
                    have_te = true;
                    pop = false;
                }
            }
        }
        if (pop) {
            if (sp == 0) break;
            --sp;
            const uint4 v = pst[sp];
            ref = v.x;
            parent = v.y >> 2;
            slot = v.y & 3u;
            m = v.z;
            have_te = false;
        }
    }
    return true;
}

// ------------------------------------------------------------------------------------------
// One traversal round over keys in (L, t_max] (Sec. III-A). With ckpt, it starts from the
// checkpoint source list (or the root in the first round), writes nodes failing the t_max
// test to the destination list and rejected hits to the eviction list (Sec. IV-B);
// otherwise it starts at the root and culls. Returns false when a capacity is exceeded.
// ------------------------------------------------------------------------------------------
template <int K, int FORM, bool INSTR>
__device__ __forceinline__ bool trace_round(const TraceArgs &a, const SceneRef &sc, float3 o, float3 d, float3 inv,
                                            float inv_len, float tn, float tf,
                                            float Lt, uint32_t Li, bool ckpt, bool from_root,
                                            uint32_t src, int n_src, uint32_t dst, int &n_dst, uint32_t ev,
                                            int &n_ev, KBuf<K> &kb, Cut &cut, int window, Counters &cnt)
{
    if constexpr (FORM == FORM_SPHERE4 || FORM == FORM_SPHERE4Q)
        return trace_round4<K, INSTR, FORM == FORM_SPHERE4Q>(a, sc, o, d, inv, tn, tf, Lt, Li, ckpt, from_root, src,
                                                             n_src, dst, n_dst, ev, n_ev, kb, cnt);
    const uint32_t S = (uint32_t)a.n_slots;
    uint2 *__restrict__ const L = a.ck0;      // lists: src, dst and ev are entry offsets into L
    // far children deferred within this round: node refs only (4 bytes each); a popped entry
    // is visited without re-testing its entry depth, since its children meet the t_max test
    uint32_t stack[GRTX_STACK];
    int sp = 0, si = 0;
    const bool windowed = FORM != FORM_PROXY && ckpt && a.window > 0;
    float tmax = windowed ? fminf(kb.n == K && n_ev >= window ? kb.tmax : GRTX_INF, cut.top(a)) : kb.tmax;
    uint32_t ref;
    float te;
    n_dst = 0;
    if (from_root) {
        n_src = 0;                    // a restart never resumes checkpointed subtrees
        ref = 0u;
        te = tn;
    } else {
        if (n_src == 0) return true;
        uint2 v = L[src];
        ref = v.x;
        te = __uint_as_float(v.y);
        si = 1;
    }
    for (;;) {
        if (te > tmax) {                              // fails the t_max test
            if (ckpt && !(windowed && te > cut.top(a))) {
                if (n_dst >= a.ckpt_cap) return false;
                L[dst + (uint32_t)n_dst * S] = make_uint2(ref, __float_as_uint(te));
                ++n_dst;
                if (INSTR) cnt.ckpt++;
            }
        } else if (INSTR && !ref_ok(sc, ref, cnt)) {  // not fetched (self-check)
        } else if (ref & GRTX_LEAF) {
            uint32_t idx = ref & ~GRTX_LEAF;
            if (INSTR) {
                cnt.leaves++;
                log_visit(cnt, ref);
            }
            uint32_t gi;
            bool touch = true;
            if (FORM == FORM_PROXY) {
                const float4 *tr = sc.tris + 3 * (size_t)idx;
                float4 v0 = __ldg(tr), v1 = __ldg(tr + 1), v2 = __ldg(tr + 2);
                gi = __float_as_uint(v0.w);
                touch = (!INSTR || gauss_ok(sc, gi, cnt)) && tri_hit(v0, v1, v2, o, d) > tn;
            } else {
                gi = idx;
                if (FORM == FORM_ICO) touch = template_touch<INSTR>(sc, gi, o, d, tn, cnt);
            }
            float t, D2, w[3];
            if (touch && sphere_test(sc.geom + 4 * (size_t)gi, o, d, t, D2, w)) {
                if (D2 <= 1.0f && t > tn && t <= tf && key_after(t, gi, Lt, Li) &&
                    !(windowed && t > cut.top(a))) {
                    if (FORM != FORM_PROXY || !kb.contains(t, gi)) {
                        float ct = t;
                        uint32_t ci = windowed ? cut.add(a, sc.geom + 4 * (size_t)gi, gi, t, D2) : gi << a.id_shift;
                        if (kb.insert(ct, ci) && ckpt) {       // any-hit: rejected -> eviction list
                            if (n_ev >= a.evict_cap) return false;
                            L[ev + (uint32_t)n_ev * S] = make_uint2(__float_as_uint(ct), ci);
                            ++n_ev;
                            if (INSTR) cnt.evictions++;
                        }
                        tmax = kb.tmax;                        // farthest kept key
                        if (windowed) tmax = fminf(n_ev >= window ? tmax : GRTX_INF, cut.top(a));
                    }
                }
            }
        } else {
            if (INSTR) {
                cnt.nodes++;
                log_visit(cnt, ref);
            }
            const float4 *nd = sc.nodes + 4 * (size_t)ref;
            float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
            uint32_t c0 = __float_as_uint(n3.x), c1 = __float_as_uint(n3.y);
            float e0, x0, e1, x1;
            slab(n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, o, inv, tn, tf, e0, x0);
            slab(n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, o, inv, tn, tf, e1, x1);
            bool h0 = e0 <= x0 && !(x0 < Lt);
            bool h1 = e1 <= x1 && !(x1 < Lt) && c1 != GRTX_NONE;
            bool near0 = e0 <= e1;
            if (FORM == FORM_PROXY) {
                // a proxy face can lie up to one proxy diameter beyond the Gaussian's key, so
                // the t_max test of a proxy subtree is taken at entry - (its largest diameter)
                e0 = fmaf(-n3.z, inv_len, e0);
                e1 = fmaf(-n3.w, inv_len, e1);
            }
            if (h0 && h1) {
                uint32_t far_ref = near0 ? c1 : c0;
                float far_t = near0 ? e1 : e0;
                ref = near0 ? c0 : c1;
                te = near0 ? e0 : e1;
                if (far_t > tmax) {
                    if (ckpt && !(windowed && far_t > cut.top(a))) {
                        if (n_dst >= a.ckpt_cap) return false;
                        L[dst + (uint32_t)n_dst * S] = make_uint2(far_ref, __float_as_uint(far_t));
                        ++n_dst;
                        if (INSTR) cnt.ckpt++;
                    }
                } else if (sp < GRTX_STACK) {
                    stack[sp++] = far_ref;
                } else if (INSTR) {
                    cnt.overflow++;
                }
                continue;
            }
            if (h0 || h1) {
                ref = h0 ? c0 : c1;
                te = h0 ? e0 : e1;
                continue;
            }
        }
        if (sp > 0) {
            ref = stack[--sp];
            te = -GRTX_INF;
        } else if (si < n_src) {
            uint2 v = L[src + (uint32_t)si * S];
            ++si;
            ref = v.x;
            te = __uint_as_float(v.y);
        } else {
            break;
        }
    }
    return true;
}

// ------------------------------------------------------------------------------------------
// A round of a warp's rays from the root as one packet (round 1, and every round when
// restarting). Every ray of a warp starts its first round at the root (Sec. III-A), and the
// rays of an 8x4 pixel tile need nearly the same nodes, so the warp
// walks one node sequence -- the union of what its rays need -- loading each node once for all
// lanes instead of once per lane, with no divergence between node and leaf steps. Each lane
// keeps its own entry test against its t_max, its k-buffer, checkpoint and eviction lists,
// exactly as in trace_round, so every ray's round ends with the same k-buffer (the traversal
// order, hence the checkpoint lists, may differ). The warp's stack (kPacketStack entries of
// (node, parent << 1 | child slot, lane mask), in shared memory) holds far children with the
// lanes that want them; a popped node's entry distance is recomputed per lane from its box in
// the parent. Every lane of the warp must call this together (full-mask ballots); lanes
// without a ray pass valid = false. lane_ok is false for a lane whose lists overflowed, and for
// every lane if the warp's stack would overflow (returns false then): such a lane redoes the
// round from the root on its own, as after any capacity overflow in trace_ray.
// ------------------------------------------------------------------------------------------
constexpr int kPacketStack = GRTX_PACKET_STACK;
constexpr unsigned kLeftCap = 1u << 18, kLeftRoom = 1u << 15;   // bundles that a launch can leave to k_trace_rays
constexpr int kDiscardRows = 64;      // see discard_dead_lists
constexpr int kWarpShared = 119;

template <int K, int FORM, bool INSTR>
__device__ __forceinline__ bool packet_round(const TraceArgs &a, const SceneRef &sc, bool valid, uint4 *pst, float3 o,
                                             float3 d, float3 inv, float inv_len, float tn, float tf, float Lt,
                                             uint32_t Li, bool ckpt, uint32_t dst, int &n_dst,
                                             uint32_t ev, int &n_ev, KBuf<K> &kb, Cut &cut, Counters &cnt,
                                             bool &lane_ok)
{
    if constexpr (FORM == FORM_SPHERE4 || FORM == FORM_SPHERE4Q)
        return packet_round4<K, INSTR, FORM == FORM_SPHERE4Q>(a, sc, valid, pst, o, d, inv, tn, tf, Lt, Li, ckpt, dst,
                                                              n_dst, ev, n_ev, kb, cnt, lane_ok);
    const unsigned full = 0xffffffffu;
    const uint32_t S = (uint32_t)a.n_slots;
    uint2 *__restrict__ const L = a.ck0;      // lists: dst and ev are entry offsets into L
    const int lane = threadIdx.x & 31;
    const bool windowed = FORM != FORM_PROXY && ckpt && a.window > 0;
    float tmax = kb.tmax;
    bool cutting = !windowed;                           // (warp-uniform) some lane has a finite t_max
    n_dst = 0;
    n_ev = 0;
    lane_ok = true;
    if (!sc.has_tree) return true;                      // nothing to traverse (uniform)
    int sp = 0;
    uint32_t ref = 0u, parent = GRTX_NONE, slot = 0u;
    unsigned m = __ballot_sync(full, valid);
    float te = tn;
    bool have_te = true;
    for (;;) {
        bool in = (m >> lane) & 1u;
        if (!have_te && !cutting) te = tn;              // no lane would fail the t_max test
        if (!have_te && cutting && in) {                // a popped node: entry from the parent's box
            const float4 *pn = sc.nodes + 4 * (size_t)parent;
            float x;
            if (slot == 0u) {
                float4 n0 = __ldg(pn), n1 = __ldg(pn + 1);
                slab(n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, o, inv, tn, tf, te, x);
            } else {
                float4 n1 = __ldg(pn + 1), n2 = __ldg(pn + 2);
                slab(n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, o, inv, tn, tf, te, x);
            }
            if (FORM == FORM_PROXY) te = fmaf(-(slot == 0u ? __ldg(pn + 3).z : __ldg(pn + 3).w), inv_len, te);
        }
        bool go = in && lane_ok && !(te > tmax);
        if (in && lane_ok && te > tmax && ckpt && !(windowed && te > cut.top(a))) {   // fails the t_max test: checkpoint it
            if (n_dst >= a.ckpt_cap) {
                lane_ok = false;
            } else {
                L[dst + (uint32_t)n_dst * S] = make_uint2(ref, __float_as_uint(te));
                ++n_dst;
                if (INSTR) cnt.ckpt++;
            }
        }
        m = __ballot_sync(full, go);
        bool pop = true;
        if (m && (!INSTR || ref_ok(sc, ref, cnt, go))) {   // ref is the warp's: all lanes agree
            if (ref & GRTX_LEAF) {
                bool touch = true;
                uint32_t gi = 0u;
                if (go) {
                    uint32_t idx = ref & ~GRTX_LEAF;
                    if (INSTR) {
                        cnt.leaves++;
                        log_visit(cnt, ref);
                    }
                    if (FORM == FORM_PROXY) {
                        const float4 *tr = sc.tris + 3 * (size_t)idx;
                        float4 v0 = __ldg(tr), v1 = __ldg(tr + 1), v2 = __ldg(tr + 2);
                        gi = __float_as_uint(v0.w);
                        touch = (!INSTR || gauss_ok(sc, gi, cnt)) && tri_hit(v0, v1, v2, o, d) > tn;
                    } else {
                        gi = idx;
                        if (FORM == FORM_ICO) touch = template_touch<INSTR>(sc, gi, o, d, tn, cnt);
                    }
                }
                // the lanes leave the template's loop at different steps and have to be told to meet
                // here: otherwise each runs the exact test alone (restart, 1M, 1280x720, 20 and 80
                // triangles: 13.8 and 20.8 ms without this, 9.9 and 11.5 with it)
                if (FORM == FORM_ICO) __syncwarp(full);
                if (go) {
                    float t, D2, w[3];
                    if (touch && sphere_test(sc.geom + 4 * (size_t)gi, o, d, t, D2, w) && D2 <= 1.0f && t > tn &&
                        t <= tf && key_after(t, gi, Lt, Li) && (FORM != FORM_PROXY || !kb.contains(t, gi)) &&
                        !(windowed && t > cut.top(a))) {
                        float ct = t;
                        uint32_t ci = windowed ? cut.add(a, sc.geom + 4 * (size_t)gi, gi, t, D2) : gi << a.id_shift;
                        if (kb.insert(ct, ci) && ckpt) {
                            if (n_ev >= a.evict_cap) {
                                lane_ok = false;
                            } else {
                                L[ev + (uint32_t)n_ev * S] = make_uint2(__float_as_uint(ct), ci);
                                ++n_ev;
                                if (INSTR) cnt.evictions++;
                            }
                        }
                        tmax = kb.tmax;
                        if (windowed) tmax = fminf(n_ev >= a.window ? tmax : GRTX_INF, cut.top(a));
                    }
                }
                if (!cutting) cutting = __any_sync(full, tmax < GRTX_INF);
            } else {
                const float4 *nd = sc.nodes + 4 * (size_t)ref;
                float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
                uint32_t c0 = __float_as_uint(n3.x), c1 = __float_as_uint(n3.y);
                bool h0 = false, h1 = false, near0 = true;
                float e0 = 0.f, e1 = 0.f;
                if (go) {
                    if (INSTR) {
                        cnt.nodes++;
                        log_visit(cnt, ref);
                    }
                    float x0, x1;
                    slab(n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, o, inv, tn, tf, e0, x0);
                    slab(n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, o, inv, tn, tf, e1, x1);
                    h0 = e0 <= x0 && !(x0 < Lt);
                    h1 = e1 <= x1 && !(x1 < Lt) && c1 != GRTX_NONE;
                    near0 = e0 <= e1;
                    if (FORM == FORM_PROXY) {             // t_max tests at entry - slack (see trace_round)
                        e0 = fmaf(-n3.z, inv_len, e0);
                        e1 = fmaf(-n3.w, inv_len, e1);
                    }
                }
                unsigned m0 = __ballot_sync(full, h0), m1 = __ballot_sync(full, h1);
                if (m0 && m1) {
                    unsigned both = m0 & m1, vote = __ballot_sync(full, h0 && h1 && near0);
                    bool n0first = both ? (2 * __popc(vote) >= __popc(both)) : (__popc(m0) >= __popc(m1));
                    if (sp >= a.packet_stack) {               // too deep for the warp's stack
                        lane_ok = false;
                        return false;
                    }
                    if (lane == 0)
                        pst[sp] = make_uint4(n0first ? c1 : c0, (ref << 1) | (n0first ? 1u : 0u), n0first ? m1 : m0, 0u);
                    ++sp;
                    __syncwarp(full);
                    parent = ref;
                    slot = n0first ? 0u : 1u;
                    m = n0first ? m0 : m1;
                    te = n0first ? e0 : e1;
                    ref = n0first ? c0 : c1;
                    have_te = true;
                    pop = false;
                } else if (m0 || m1) {
                    parent = ref;
                    slot = m0 ? 0u : 1u;
                    m = m0 ? m0 : m1;
                    te = m0 ? e0 : e1;
                    ref = m0 ? c0 : c1;
                    have_te = true;
                    pop = false;
                }
            }
        }
        if (pop) {
            if (sp == 0) break;
            --sp;
            uint4 v = pst[sp];
            ref = v.x;
            parent = v.y >> 1;
            slot = v.y & 1u;
            m = v.z;
            have_te = false;
        }
    }
    return true;
}

// ------------------------------------------------------------------------------------------
// The first round of a warp's rays over sphere leaves, walked for the tile instead of for each
// ray. The warp bounds its rays by the box of their origins and the box of their directions, and
// each lane takes one pending node and tests the node's two child boxes against that bundle, so
// that one step expands up to 32 nodes. Leaves are gathered and tested in groups of 32: first
// every ray filters all 32 (one broadcast record load each), which gives each lane a mask of its
// candidates; then each lane takes its own candidates one after another through the exact test.
// The k-buffer, eviction list and Cut of each ray are those of trace_round; there are no
// checkpoints (a ray whose eviction list is too small leaves the walk and takes trace_round).
//
// Why: a packet that tests one node at a time for 32 rays is a chain of about 340 node steps, 150
// pops and 130 leaf steps a tile on the 1M surface frame, and its exact tests run with a quarter
// of the lanes. The walk takes 27 steps, 145 filters and 51 exact tests with 23 lanes each:
// 2.6 G instead of 7.8 G warp instructions a frame. 1920x1080, k = 16: 9.8 ms with packets and
// per-ray later rounds, 6.8 ms with packets bounded by opacity (Cut), 3.9 ms with the walk, 3.5 with
// the quadratic filter below, 3.2 with 64-bit keys and 256-bit gathers. What bounds it now: the L1
// pipe (80 %: each lane gathers its own records and SH coefficients) and instruction issue (68 %).
// Keeping the hits' alphas instead of testing again at the blend, colours by groups of four lanes, and
// 5 to 7 blocks an SM with the registers for it were measured: none was faster.
// Groups of 8 or 16 rays with a stack each took 7.9 and 4.7 ms against 4.0 for one of 32.
// ------------------------------------------------------------------------------------------
// The stack keeps a quarter of its entries for walking one node at a time: past three quarters of
// pending nodes a step takes the top one only, as a depth-first walk does. It has four entries for each
// of a packet's (with as many as a packet's, packet_stack = 24 took a 640x360 frame of 1M Gaussians 3.1
// instead of 1.75 ms, 200,000 scattered rays 11.9 instead of 3.95 ms, and these with 8 14.0 instead of 5.5).
// (A stack of 128 with 96 leaves: preview 847 instead of 556 us, since wide tiles then walk node by
// node; 96 leaves with this stack: frame +1 %.)
constexpr int kWalkStack = 4 * kPacketStack, kWalkLeaves = 128;

struct __align__(16) WalkShared {
    uint32_t stack[kWalkStack];  // pending nodes
    uint32_t leaf[kWalkLeaves];  // gathered leaves
    float c[12];                 // per axis: origin max, 1 / direction max, origin min, 1 / direction min
    float mid[4];                // middle of the direction box, and the largest distance of a ray's direction from it
    int rows;                    // of the eviction lists that the walk's rays filled, or -1 if rays went on per ray
    int pad;
    uint2 place;                 // what the bundle's entry in the left list would be
    float4 off[32];              // each ray's direction minus mid (rays of one origin)
};

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}

// Checks of a checked walk: the pending node at entry e of the stack; the leaf slots among a node's
// children.
template <bool CHK>
__device__ __forceinline__ bool next_node(const TraceArgs &a, const SceneRef &sc, const WalkShared &w, int e)
{
    return !CHK || (in_bounds<CHK>(a, (uint32_t)e, kWalkStack) && in_bounds<CHK>(a, w.stack[e], sc.n_nodes));
}
__device__ __forceinline__ void drop_bad_leaves(const TraceArgs &a, const SceneRef &sc, uint32_t &c0, uint32_t &c1)
{
    if (c0 != GRTX_NONE && (c0 & GRTX_LEAF) && !in_bounds<true>(a, c0 & ~GRTX_LEAF, sc.n_geom)) c0 = GRTX_NONE;
    if (c1 != GRTX_NONE && (c1 & GRTX_LEAF) && !in_bounds<true>(a, c1 & ~GRTX_LEAF, sc.n_geom)) c1 = GRTX_NONE;
}

// One axis of the bundle test. A ray of the bundle is inside [lo, hi] on this axis at depth t only
// if lo <= o_max + t d_max and hi >= o_min + t d_min; each condition bounds t from below or from
// above, by the sign of its direction bound (c[1], c[3] hold the reciprocals).
__device__ __forceinline__ void bundle_axis(const float *c, float lo, float hi, float &e, float &x)
{
    const float ra = c[1], rb = c[3];
    const float ta = (lo - c[0]) * ra, tb = (hi - c[2]) * rb;
    if (ra > 0.f) e = fmaxf(e, ta); else x = fminf(x, ta);
    if (rb > 0.f) x = fminf(x, tb); else e = fmaxf(e, tb);
}

// Shortens a ray's eviction list (n entries, row stride S) in the walk. Where the k-buffer and the
// entries up to the list's mean depth m already hold the opacity at which the ray ends (need, in
// bits, from the entries' codes), nothing behind m can be blended: m becomes the ray's end (end =
// true). Otherwise, with full set, m becomes the limit of this round (the ray's later rounds start
// behind it, see trace_ray). Either way the entries behind m are dropped. Returns m, or +inf where
// the list stays as it is.
template <int K>
static __device__ __noinline__ float squeeze(uint2 *L, uint32_t S, int n, int &kept, const uint64_t *keys,
                                             float need, bool full, bool &end)
{
    float sum = 0.f;
#pragma unroll 4
    for (int e = 0; e < n; ++e) sum += __uint_as_float(L[(uint32_t)e * S].x);
    const float m = fmaxf(sum / (float)n, depth_of_key(keys[(K - 1) * kBlock]));       // entries in the k-buffer stay within it
    float bits = 0.f;
#pragma unroll
    for (int j = 0; j < K; ++j) bits += opacity_of_code((uint32_t)keys[j * kBlock] & ((1u << kCodeBits) - 1u));
#pragma unroll 4
    for (int e = 0; e < n; ++e) {
        const uint2 v = L[(uint32_t)e * S];
        if (!(__uint_as_float(v.x) > m)) bits += opacity_of_code(v.y & ((1u << kCodeBits) - 1u));
    }
    end = bits > need;
    kept = n;
    if (!end && !full) return GRTX_INF;
    int k = 0;
    for (int e = 0; e < n; ++e) {
        const uint2 v = L[(uint32_t)e * S];
        if (!(__uint_as_float(v.x) > m)) {
            L[(uint32_t)k * S] = v;
            ++k;
        }
    }
    kept = k;
    return m;
}

// Entries a list may grow by before it is squeezed: 48 / 64 / 96 gave 3.28 / 3.25 / 3.22 ms for the
// 1M 1080p frame (few rays ever do) and 12.0 / 11.8 / 12.2 ms for the 6M outdoor frame (fog).
constexpr int kSqueeze = 64;
// Work (in leaf tests; a step counts as 4) after which a walk with fewer than one candidate per
// four is given up: its rays share almost nothing, and each traces the round on its own. Given up
// after 128 / 256 / 512 / 1024, the 256x256 preview took 860 / 725 / 604 / 604 us (its wide tiles are
// still far cheaper than rays on their own) and the 1080p frame 4.24 / 3.47 / 3.47 / 3.47 ms.
// The work of rays of several origins that can be left to k_trace_rays (ray lists) counts double, since
// the one-ray kernel costs them less, and a lone list leaves a bundle after kListWork of it whatever it
// shares: the few bundles deep in fog are the launch's last, and go faster a ray to a warp. 70,354 bounce
// rays over 6M Gaussians in bundles of 8, k = 16 / 32: neither 4.8 / 4.9 ms, counted double 4.4 / 3.5, left
// after 1024 / 2048 / 3072 / 4096 / 6144 of it 3.6 / 3.36 / 3.4 / 3.9 / 4.1 ms (k = 16). In a batch the
// one-ray kernel would begin only behind the images: 11.4 ms without kListWork, 11.6 with it.
constexpr int kWalkTrial = 512, kListWork = 2048;

// Which rays of one origin o may hit a Gaussian, as one quadratic in the ray's direction. A ray
// d = mid + x meets the Gaussian where |o_l x d_l|^2 <= |d_l|^2 (o_l = A (o - mu), d_l = A d): with
// c0 = o_l x A mid and the columns a_k of A, C_k = o_l x a_k, that is
//   |c0|^2 - |A mid|^2 + sum_k 2 (c0.C_k - A mid.a_k) x_k + sum_kl (C_k.C_l - a_k.a_l) x_k x_l <= 0,
// divided by |A mid|^2. Each lane sets up one leaf (about 150 instructions), then every ray costs 9
// FMAs a leaf instead of the 45 of sphere_candidate. The test only filters, so it is widened by its
// rounding: |o_l| and d_l err by up to e = 2e-6 |A| |o - mu| in units of the sphere (taken as 32 ulp
// of the products), and the sum by 2e-6 of its largest terms: c0, the C_k and the a_k over the
// tile's radius r (the last weigh most where the middle ray lies in a thin Gaussian's plane).
struct ConeTest {
    float c, bx, by, bz, xx, yy, zz, xy, xz, yz;
    __device__ __forceinline__ void set(float4 r0, float4 r1, float4 r2, float3 o, float3 m, float r)
    {
        const float vx = o.x - r0.w, vy = o.y - r1.w, vz = o.z - r2.w;
        const float o0 = r0.x * vx + r0.y * vy + r0.z * vz, o1 = r1.x * vx + r1.y * vy + r1.z * vz,
                    o2 = r2.x * vx + r2.y * vy + r2.z * vz;
        const float d0 = r0.x * m.x + r0.y * m.y + r0.z * m.z, d1 = r1.x * m.x + r1.y * m.y + r1.z * m.z,
                    d2 = r2.x * m.x + r2.y * m.y + r2.z * m.z;
        const float inv = 1.0f / (d0 * d0 + d1 * d1 + d2 * d2);
        const float t = -(o0 * d0 + o1 * d1 + o2 * d2) * inv;
        const float p0 = fmaf(t, d0, o0), p1 = fmaf(t, d1, o1), p2 = fmaf(t, d2, o2);
        // c0 = p x d_l: the part of o_l along A mid drops out
        const float c0 = p1 * d2 - p2 * d1, c1 = p2 * d0 - p0 * d2, c2 = p0 * d1 - p1 * d0;
        const float X0 = o1 * r2.x - o2 * r1.x, X1 = o2 * r0.x - o0 * r2.x, X2 = o0 * r1.x - o1 * r0.x;
        const float Y0 = o1 * r2.y - o2 * r1.y, Y1 = o2 * r0.y - o0 * r2.y, Y2 = o0 * r1.y - o1 * r0.y;
        const float Z0 = o1 * r2.z - o2 * r1.z, Z1 = o2 * r0.z - o0 * r2.z, Z2 = o0 * r1.z - o1 * r0.z;
        const float axx = r0.x * r0.x + r1.x * r1.x + r2.x * r2.x, ayy = r0.y * r0.y + r1.y * r1.y + r2.y * r2.y,
                    azz = r0.z * r0.z + r1.z * r1.z + r2.z * r2.z;
        const float e = 2e-6f * sqrtf((axx + ayy + azz) * (vx * vx + vy * vy + vz * vz)), g = 1.0f + 2.0f * e + e * e;
        const float Xx = X0 * X0 + X1 * X1 + X2 * X2, Yy = Y0 * Y0 + Y1 * Y1 + Y2 * Y2, Zz = Z0 * Z0 + Z1 * Z1 + Z2 * Z2;
        const float cc = (c0 * c0 + c1 * c1 + c2 * c2) * inv;
        c = cc - g - 2e-6f * (cc + r * r * (Xx + Yy + Zz + g * (axx + ayy + azz)) * inv + g);
        bx = 2.0f * inv * (c0 * X0 + c1 * X1 + c2 * X2 - g * (d0 * r0.x + d1 * r1.x + d2 * r2.x));
        by = 2.0f * inv * (c0 * Y0 + c1 * Y1 + c2 * Y2 - g * (d0 * r0.y + d1 * r1.y + d2 * r2.y));
        bz = 2.0f * inv * (c0 * Z0 + c1 * Z1 + c2 * Z2 - g * (d0 * r0.z + d1 * r1.z + d2 * r2.z));
        xx = inv * (Xx - g * axx);
        yy = inv * (Yy - g * ayy);
        zz = inv * (Zz - g * azz);
        xy = 2.0f * inv * (X0 * Y0 + X1 * Y1 + X2 * Y2 - g * (r0.x * r0.y + r1.x * r1.y + r2.x * r2.y));
        xz = 2.0f * inv * (X0 * Z0 + X1 * Z1 + X2 * Z2 - g * (r0.x * r0.z + r1.x * r1.z + r2.x * r2.z));
        yz = 2.0f * inv * (Y0 * Z0 + Y1 * Z1 + Y2 * Z2 - g * (r0.y * r0.z + r1.y * r1.z + r2.y * r2.z));
    }
    __device__ __forceinline__ bool miss(float4 x) const
    {
        const float a = fmaf(xz, x.z, fmaf(xy, x.y, fmaf(xx, x.x, bx)));
        const float b = fmaf(yz, x.z, fmaf(yy, x.y, by)), d = fmaf(zz, x.z, bz);
        return fmaf(d, x.z, fmaf(b, x.y, fmaf(a, x.x, c))) > 0.f;
    }
};

// Walks the bundle of the warp's valid rays (the other lanes help, and keep their rays' state).
// lane_ok becomes false for a ray whose eviction list was too small. Returns false if the bundle was
// left: no stack, a ray that cannot be bounded, or too little shared. base: added to the leaf slots
// (a world's objects; the state of the rays goes on from call to call).
template <int K, bool CHK = false>
__device__ __forceinline__ bool tile_walk(const TraceArgs &a, const SceneRef &sc, bool valid, WalkShared &w,
                                          float3 o, float3 d, float tn, float tf, uint32_t ev, int &n_ev, KBuf<K> &kb,
                                          Cut &cut, float &lim, bool &lane_ok, uint32_t base = 0u)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t S = (uint32_t)a.n_slots;
    uint2 *__restrict__ const L = a.ck0;
    if (!__any_sync(full, valid)) return true;
    // a ray that is not finite cannot be bounded, and a bundle bounds depths from 0 on
    const bool odd = valid && !(fabsf(o.x) + fabsf(o.y) + fabsf(o.z) + fabsf(d.x) + fabsf(d.y) + fabsf(d.z) < 3e38f && tn >= 0.f);
    if (__any_sync(full, odd)) return false;
    const float t0 = warp_min(valid ? tn : GRTX_INF);
    float tile_max = warp_max(valid ? tf : 0.f);     // no ray of the bundle needs anything beyond
    bool one_origin = true, every_way = true;
    {
        // bounds of the bundle; a direction bound of 0 is moved outwards to keep its reciprocal finite
        const float oc[3] = {o.x, o.y, o.z}, dc[3] = {d.x, d.y, d.z};
        float mid[3];
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float omax = warp_max(valid ? oc[q] : -GRTX_INF), omin = warp_min(valid ? oc[q] : GRTX_INF);
            float dmax = warp_max(valid ? dc[q] : -GRTX_INF), dmin = warp_min(valid ? dc[q] : GRTX_INF);
            mid[q] = 0.5f * dmin + 0.5f * dmax;
            one_origin = one_origin && omin == omax;
            every_way = every_way && dmin < 0.f && dmax > 0.f;
            if (fabsf(dmax) < 1e-30f) dmax = 1e-30f;
            if (fabsf(dmin) < 1e-30f) dmin = -1e-30f;
            if (lane == 0) {
                w.c[4 * q] = omax;
                w.c[4 * q + 1] = 1.0f / dmax;
                w.c[4 * q + 2] = omin;
                w.c[4 * q + 3] = 1.0f / dmin;
            }
        }
        if (every_way) return false;         // the direction box holds 0: it bounds nothing
        const float4 x = valid ? make_float4(d.x - mid[0], d.y - mid[1], d.z - mid[2], 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float r = sqrtf(warp_max(x.x * x.x + x.y * x.y + x.z * x.z));
        w.off[lane] = x;
        if (lane == 0) {
            w.stack[0] = 0u;
            w.mid[0] = mid[0];
            w.mid[1] = mid[1];
            w.mid[2] = mid[2];
            w.mid[3] = r;
        }
        __syncwarp();
    }
    const int cap = a.packet_stack * (kWalkStack / kPacketStack), wide = cap - cap / 4;
    const int unit = a.left && !one_origin ? 2 : 1, most = unit == 2 ? a.leave_at : 0x7fffffff;      // (see kWalkTrial)
    int sp = 1, nl = 0, work = 0, cands = 0;
    int squeeze_at = min(kSqueeze, max(a.evict_cap - 31, 1));
    for (;;) {
        // expand up to 32 pending nodes, nearest first (lane 0 takes the top of the stack)
        if (sp >= cap || (work >= kWalkTrial && (4 * cands < work || work >= most))) return false;   // no room, or too little shared
        const int p = min(min(32, sp), max(1, wide - sp));
        uint32_t cn = GRTX_NONE, cf = GRTX_NONE;                     // near and far child to visit
        if (lane < p && next_node<CHK>(a, sc, w, sp - 1 - lane)) {
            const float4 *nd = sc.nodes + 4 * (size_t)w.stack[sp - 1 - lane];
            float4 n0, n1, n2, n3;
            ldg2(nd, n0, n1);
            ldg2(nd + 2, n2, n3);
            float e0 = t0, x0 = tile_max, e1 = t0, x1 = tile_max;
            bundle_axis(w.c, n0.x, n0.w, e0, x0);
            bundle_axis(w.c + 4, n0.y, n1.x, e0, x0);
            bundle_axis(w.c + 8, n0.z, n1.y, e0, x0);
            bundle_axis(w.c, n1.z, n2.y, e1, x1);
            bundle_axis(w.c + 4, n1.w, n2.z, e1, x1);
            bundle_axis(w.c + 8, n2.x, n2.w, e1, x1);
            // the bounds are rounded: an entry is lowered by 4e-6 of its depth, far more than its rounding
            cn = e0 * (1.0f - 4e-6f) <= x0 ? __float_as_uint(n3.x) : GRTX_NONE;
            cf = e1 * (1.0f - 4e-6f) <= x1 ? __float_as_uint(n3.y) : GRTX_NONE;
            if (e1 < e0) {
                const uint32_t t = cn; cn = cf; cf = t;
            }
            if (CHK) drop_bad_leaves(a, sc, cn, cf);
        }
        __syncwarp();
        const bool ln = cn != GRTX_NONE && (cn & GRTX_LEAF), lf = cf != GRTX_NONE && (cf & GRTX_LEAF);
        const unsigned bn = __ballot_sync(full, cn != GRTX_NONE && !ln), bf = __ballot_sync(full, cf != GRTX_NONE && !lf);
        const unsigned gn = __ballot_sync(full, ln), gf = __ballot_sync(full, lf);
        const unsigned below = (1u << lane) - 1u, above = ~(below | (1u << lane));
        sp -= p;
        work += 4 * unit;
        int at = sp + __popc(bn & above) + __popc(bf & above);
        if (cf != GRTX_NONE && !lf && in_bounds<CHK>(a, at, kWalkStack)) w.stack[at++] = cf;
        if (cn != GRTX_NONE && !ln && in_bounds<CHK>(a, at, kWalkStack)) w.stack[at] = cn;
        sp += __popc(bn) + __popc(bf);
        at = nl + __popc(gn & below) + __popc(gf & below);
        if (ln && in_bounds<CHK>(a, at, kWalkLeaves)) w.leaf[at++] = cn & ~GRTX_LEAF;
        if (lf && in_bounds<CHK>(a, at, kWalkLeaves)) w.leaf[at] = cf & ~GRTX_LEAF;
        nl += __popc(gn) + __popc(gf);
        __syncwarp();
        if (sp > 0 && nl <= kWalkLeaves - 64) continue;
        // test the gathered leaves, 32 at a time: a mask of the ray's candidates, ...
        for (int g0 = 0; g0 < nl; g0 += 32) {
            const int m = min(32, nl - g0);
            unsigned mask = 0;
            const float bound = fminf(fminf(tf, lim), cut.top(a));
            if (one_origin) {
                // a lane takes a leaf and goes through the rays
                const float4 *g = sc.geom + 4 * (size_t)w.leaf[g0 + min(lane, m - 1)];
                ConeTest q;
                const float3 oo = make_float3(w.c[0], w.c[4], w.c[8]);
                float4 r0, r1, r2, r3;
                ldg2(g, r0, r1);
                ldg2(g + 2, r2, r3);
                q.set(r0, r1, r2, oo, make_float3(w.mid[0], w.mid[1], w.mid[2]), w.mid[3]);
                const unsigned rays = __ballot_sync(full, valid);
                for (int r0 = 0; rays >> r0; r0 += 8) {
#pragma unroll
                    for (int r = r0; r < r0 + 8; ++r) {
                        const unsigned b = __ballot_sync(full, !q.miss(w.off[r]));
                        if (lane == r) mask = b;
                    }
                    if (r0 == 24) break;
                }
                mask &= m == 32 ? full : (1u << m) - 1u;
            } else {
                for (int i = 0; i < m; ++i) {
                    const float4 *g = sc.geom + 4 * (size_t)w.leaf[g0 + i];
                    float t, aa;
                    if (sphere_candidate(__ldg(g), __ldg(g + 1), __ldg(g + 2), o, d, t, aa) && in_range(t, aa, tn, bound))
                        mask |= 1u << i;
                }
            }
            if (!(valid && lane_ok)) mask = 0;
            work += m * unit;
            cands += __reduce_add_sync(full, __popc(mask));
            // ... then the candidates of each ray one after another
            while (mask) {
                const int i = __ffs(mask) - 1;
                mask &= mask - 1u;
                const uint32_t gi = w.leaf[g0 + i];
                const float4 *g = sc.geom + 4 * (size_t)gi;
                float t, D2, u[3], aa;
                float4 r0, r1, r2, r3;
                ldg2(g, r0, r1);
                ldg2(g + 2, r2, r3);
                if (!sphere_candidate(r0, r1, r2, o, d, t, aa) || !in_range(t, aa, tn, fminf(bound, cut.top(a)))) continue;
                sphere_refine(r0, r1, r2, o, d, t, D2, u);
                if (D2 <= 1.0f && t > tn && t <= tf && !(t > fminf(lim, cut.top(a)))) {
                    float ct = t;
                    uint32_t ci = cut.take(a, 1.0f - fminf(r3.x * exp2f(r3.y * D2), a.alpha_max), base + gi, t);
                    if (kb.insert(ct, ci)) {
                        if (n_ev >= a.evict_cap) {
                            lane_ok = false;
                            break;
                        }
                        if (in_bounds<CHK>(a, n_ev, a.evict_cap)) L[ev + (uint32_t)n_ev * S] = make_uint2(__float_as_uint(ct), ci);
                        ++n_ev;
                    }
                }
            }
            __syncwarp();
            // long lists: find each ray's end, or make room for the next group (rays that are nearly due
            // take part, so that the warp does this seldom)
            if (__any_sync(full, n_ev >= squeeze_at)) {
                if (4 * n_ev >= 3 * squeeze_at && lane_ok) {
                    const bool no_room = n_ev + 32 > a.evict_cap;
                    bool end;
                    const float to = squeeze<K>(L + ev, S, n_ev, n_ev, kb.k,
                                                a.id_shift && a.p_stop > 0.f ? -__log2f(a.p_stop) : GRTX_INF, no_room, end);
                    if (end) {
                        cut.P = 0.f;
                        cut.far = to;
                    } else if (no_room) {
                        lim = to;
                    }
                    squeeze_at = min(n_ev + kSqueeze, max(a.evict_cap - 31, 1));
                }
                __syncwarp();
            }
            const float need = valid && lane_ok ? fmaxf(fminf(fminf(tf, lim), cut.top(a)), 0.f) : 0.f;
            tile_max = __uint_as_float(__reduce_max_sync(full, __float_as_uint(need)));
        }
        nl = 0;
        if (sp == 0) return true;
    }
}

// ------------------------------------------------------------------------------------------
// Blending (Sec. II-B Eq. volume-render) and its derivative.
// ------------------------------------------------------------------------------------------
struct BlendState {
    float C[3];
    float T;
    // backward
    float G[4];        // dL/d(r, g, b, T_out)
    float Cf[3];       // forward colour without background
    float Tf;          // forward transmittance at termination
    float dLdT;        // dL/dT_out + bg . dL/dC
};

__device__ __forceinline__ float atomic_add_f(float *p, float v)
{
    return atomicAdd(p, v);
}

// alpha and colour of leaf slot idx on a ray, as the forward blend_one computes them.
__device__ __forceinline__ float blend_terms(const TraceArgs &a, const SceneRef &sc, uint32_t idx, float3 o, float3 d, float c[3])
{
    const float nrm = rsqrtf(d.x * d.x + d.y * d.y + d.z * d.z);
    const float4 *g = sc.geom + 4 * (size_t)idx;
    const float4 r0 = __ldg(g), r1 = __ldg(g + 1), r2 = __ldg(g + 2), r3 = __ldg(g + 3);
    float t, D2, e[3], raw[3], Y[16];
    sphere_candidate(r0, r1, r2, o, d, t);
    sphere_refine(r0, r1, r2, o, d, t, D2, e);
    sh_color(sc.app + (size_t)idx * sc.app_stride, sc.sh_degree, sc.app_stride,
             make_float3(d.x * nrm, d.y * nrm, d.z * nrm), c, raw, Y);
    const float al = r3.x * exp2f(r3.y * D2);
    return al < a.alpha_max ? al : a.alpha_max;
}

template <bool BWD>
__device__ __forceinline__ void blend_one(const TraceArgs &a, const SceneRef &sc, BlendState &st, uint32_t idx,
                                          float3 o, float3 d)
{
    const float nrm = rsqrtf(d.x * d.x + d.y * d.y + d.z * d.z);     // colour along the unit direction
    const float3 dn = make_float3(d.x * nrm, d.y * nrm, d.z * nrm);
    const float4 *g = sc.geom + 4 * (size_t)idx;
    float t, D2, e[3];
    float4 r3;
    {
        float4 r0, r1, r2;
        ldg2(g, r0, r1);
        ldg2(g + 2, r2, r3);
        sphere_candidate(r0, r1, r2, o, d, t);
        sphere_refine(r0, r1, r2, o, d, t, D2, e);
    }
    float al_raw = r3.x * exp2f(r3.y * D2);
    bool clamped = !(al_raw < a.alpha_max);
    float al = clamped ? a.alpha_max : al_raw;
    float c[3], raw[3], Y[16];
    sh_color<BWD>(sc.app + (size_t)idx * sc.app_stride, sc.sh_degree, sc.app_stride, dn, c, raw, Y);
    float w = st.T * al;
    if (!BWD) {
        st.C[0] = fmaf(w, c[0], st.C[0]);
        st.C[1] = fmaf(w, c[1], st.C[1]);
        st.C[2] = fmaf(w, c[2], st.C[2]);
        st.T *= (1.0f - al);
        return;
    }
    uint32_t gi = sc.gid[idx];
    // colour: dC/dc = T alpha; c = max(0, raw)
    if (a.g_sh) {
        const float dc[3] = {raw[0] > 0.f ? st.G[0] * w : 0.f, raw[1] > 0.f ? st.G[1] * w : 0.f,
                             raw[2] > 0.f ? st.G[2] * w : 0.f};
        float *gs = a.g_sh + (size_t)gi * a.n_sh;
        if (a.vec_sh) {
            // degree 3: the 48 coefficient gradients as 12 vector atomics (sm_90+ float4 add)
            if (dc[0] != 0.f || dc[1] != 0.f || dc[2] != 0.f) {
#pragma unroll
                for (int j = 0; j < 12; ++j) {
                    float v[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[e] = Y[(4 * j + e) / 3] * dc[(4 * j + e) % 3];
                    atomicAdd(reinterpret_cast<float4 *>(gs) + j, make_float4(v[0], v[1], v[2], v[3]));
                }
            }
        } else {
            int nk = (sc.sh_degree + 1) * (sc.sh_degree + 1);
            for (int ch = 0; ch < 3; ++ch) {
                if (dc[ch] == 0.f) continue;
                for (int k = 0; k < nk; ++k) atomic_add_f(gs + 3 * k + ch, dc[ch] * Y[k]);
            }
        }
    }
    st.C[0] = fmaf(w, c[0], st.C[0]);
    st.C[1] = fmaf(w, c[1], st.C[1]);
    st.C[2] = fmaf(w, c[2], st.C[2]);
    float inv1m = __fdividef(1.0f, 1.0f - al);           // 1 - al >= 1 - alpha_max > 0
    float dLda = -st.dLdT * st.Tf * inv1m;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) dLda += st.G[ch] * (st.T * c[ch] - (st.Cf[ch] - st.C[ch]) * inv1m);
    st.T *= (1.0f - al);
    if (clamped || dLda == 0.f) return;
    if (!a.g_stage) return;
    // alpha = o exp(-d2/2), d2 = |S^-1 R^T (x* - mu)|^2 at x* = o + t d (t fixed: envelope).
    // The raw parameters come packed in leaf order, (mu, logit), (log-scales, 0), q.
    const float4 *rw = sc.raw + 3 * (size_t)idx;
    const float4 r_ml = __ldg(rw), r_ls = __ldg(rw + 1), r_q = __ldg(rw + 2);
    float op = __fdividef(1.0f, 1.0f + expf(-r_ml.w));
    const float g_logit = dLda * al_raw * (1.0f - op);
    float dLdd2 = -0.5f * dLda * al_raw;
    // inverse scales 1/s_j = exp(-log s_j)
    float is[3] = {expf(-r_ls.x), expf(-r_ls.y), expf(-r_ls.z)};
    float qw = r_q.x, qx = r_q.y, qy = r_q.z, qz = r_q.w;
    float iq = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
    float w_ = qw * iq, x = qx * iq, y = qy * iq, z = qz * iq;
    float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w_ * z), 2.f * (x * z + w_ * y)},
                     {2.f * (x * y + w_ * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w_ * x)},
                     {2.f * (x * z - w_ * y), 2.f * (y * z + w_ * x), 1.f - 2.f * (x * x + y * y)}};
    float v[3], vs[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        float u = R[0][j] * e[0] + R[1][j] * e[1] + R[2][j] * e[2];
        v[j] = u * is[j];
        vs[j] = v[j] * is[j];
    }
    float gm[3];
#pragma unroll
    for (int c2 = 0; c2 < 3; ++c2) gm[c2] = -2.0f * dLdd2 * (R[c2][0] * vs[0] + R[c2][1] * vs[1] + R[c2][2] * vs[2]);
    // staged per leaf (three vector atomics); added into the caller's arrays after the kernel
    float4 *stage = a.g_stage + 3 * (size_t)idx;
    atomicAdd(stage, make_float4(gm[0], gm[1], gm[2], g_logit));
    atomicAdd(stage + 1, make_float4(-2.0f * dLdd2 * v[0] * v[0], -2.0f * dLdd2 * v[1] * v[1],
                                     -2.0f * dLdd2 * v[2] * v[2], 0.f));
    {
        float Gr[3][3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < 3; ++j) Gr[r][j] = 2.0f * dLdd2 * vs[j] * e[r];
        float gw = 2.f * (-z * Gr[0][1] + y * Gr[0][2] + z * Gr[1][0] - x * Gr[1][2] - y * Gr[2][0] + x * Gr[2][1]);
        float gx = 2.f * (y * Gr[0][1] + z * Gr[0][2] + y * Gr[1][0] - 2.f * x * Gr[1][1] - w_ * Gr[1][2] +
                          z * Gr[2][0] + w_ * Gr[2][1] - 2.f * x * Gr[2][2]);
        float gy = 2.f * (-2.f * y * Gr[0][0] + x * Gr[0][1] + w_ * Gr[0][2] + x * Gr[1][0] + z * Gr[1][2] -
                          w_ * Gr[2][0] + z * Gr[2][1] - 2.f * y * Gr[2][2]);
        float gz = 2.f * (-2.f * z * Gr[0][0] - w_ * Gr[0][1] + x * Gr[0][2] + w_ * Gr[1][0] - 2.f * z * Gr[1][1] +
                          y * Gr[1][2] + x * Gr[2][0] + y * Gr[2][1]);
        float dot = w_ * gw + x * gx + y * gy + z * gz;
        atomicAdd(stage + 2, make_float4((gw - w_ * dot) * iq, (gx - x * dot) * iq, (gy - y * dot) * iq,
                                         (gz - z * dot) * iq));
    }
}

// ------------------------------------------------------------------------------------------
// One ray: the round loop of Listing 1's raygen shader. PASS: the forward, the backward (same
// rounds, gradients while blending), or the forward that also saves each ray's blend list.
// ------------------------------------------------------------------------------------------
enum { PASS_FWD = 0, PASS_BWD = 1, PASS_SAVE = 2 };

// Blend-list entry j of a ray whose forward saved its list, and the end of its list.
__device__ __forceinline__ void save_blended(const TraceArgs &a, int64_t pix, int j, uint32_t idx)
{
    if (j < a.save_cap) a.save_leaves[(size_t)pix * a.save_cap + j] = idx;
}

constexpr int kMeetLists = 64;

template <int K, int FORM, bool INSTR, int PASS, bool MEET = true>
__device__ __forceinline__ void trace_ray(const TraceArgs &a, const SceneRef &sc, float4 *__restrict__ out, int slot,
                                          int64_t pix, float3 o, float3 d, float tn, float tf, KBuf<K> &kb,
                                          Counters &cnt, Cut cut, unsigned live, bool r1_done = false, bool r1_ok = true,
                                          int r1_n_dst = 0, int r1_n_ev = 0, float lim = INFINITY)
{
    constexpr bool BWD = PASS == PASS_BWD;
    const uint32_t S = (uint32_t)a.n_slots;
    float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    const float inv_len = rsqrtf(d.x * d.x + d.y * d.y + d.z * d.z);
    BlendState st;
    st.C[0] = st.C[1] = st.C[2] = 0.f;
    st.T = 1.f;
    if (BWD) {
        float4 F = a.fwd_rgbT[pix], G = a.dL_drgbT[pix];
        st.G[0] = G.x; st.G[1] = G.y; st.G[2] = G.z; st.G[3] = G.w;
        st.Tf = F.w;
        st.Cf[0] = F.x - F.w * a.bg0;
        st.Cf[1] = F.y - F.w * a.bg1;
        st.Cf[2] = F.z - F.w * a.bg2;
        st.dLdT = G.w + a.bg0 * G.x + a.bg1 * G.y + a.bg2 * G.z;
    }
    float Lt = tn;
    uint32_t Li = GRTX_NONE;
    bool ckpt = a.traversal == GRTX_TRAVERSAL_CHECKPOINT;
    bool from_root = true;
    int n_src = 0, n_ev = 0, nb = 0;
    uint32_t src = (uint32_t)slot, dst = a.ck1_off + (uint32_t)slot;      // entry offsets into a.ck0
    const uint32_t ev = a.ev_off + (uint32_t)slot;
    bool done = !sc.has_tree;
    bool first_round = true;
    // The lanes of `live` (the caller's mask of this call) meet behind each round's traversal. It has several
    // ways out, and left to the compiler the lanes that restart, which run a copy of it, may do so one after
    // another: 640x360 of 1M Gaussians with eviction lists of 16 / 40: 3.38 / 2.68 ms, 5.3 / 3.2 without; 1M / 6M
    // 1080p frame over 4-wide nodes 9.8 / 16.9 ms, 9.8 / 19.5 without. (In one copy, round the loop again: 3.45 /
    // 2.76 and 10.7 / 16.0 ms, and small frames at k = 32 5 % slower.) The frame kernel, whose rays hardly
    // ever restart with lists of 64 entries or more, leaves it out for these (!MEET): 256x256 preview 554
    // instead of 561 us, 1080p frame 3.60 instead of 3.62 ms; the server's spills more with the choice.
    const bool meet = MEET || a.evict_cap < kMeetLists;
    for (;;) {
        if (meet) live = __ballot_sync(live, !done);
        if (done) break;
        if (INSTR) cnt.rounds++;
        if (!(r1_done && first_round)) kb.clear();
        if (ckpt && n_ev > 0) {            // raygen: closest evicted hits -> k-buffer
            int w = 0;
            for (int e = 0; e < n_ev; ++e) {
                uint2 v = a.ck0[ev + (uint32_t)e * S];
                float ct = __uint_as_float(v.x);
                uint32_t ci = v.y;
                // the proxy form can find one Gaussian through several triangles, so an evicted
                // copy may already be blended (key <= L) or already be in the buffer
                if (FORM == FORM_PROXY && (!key_after(ct, ci, Lt, Li) || kb.contains(ct, ci))) continue;
                if (kb.insert(ct, ci)) {
                    a.ck0[ev + (uint32_t)w * S] = make_uint2(__float_as_uint(ct), ci);
                    ++w;
                }
            }
            n_ev = w;
        }
        int n_dst = 0;
        bool round_ok;
        if (r1_done && first_round) {                  // round 1 was traced for the warp
            round_ok = r1_ok;
            n_dst = r1_n_dst;
            n_ev = r1_n_ev;
        } else {
            round_ok = trace_round<K, FORM, INSTR>(a, sc, o, d, inv, inv_len, tn, tf, Lt, Li, ckpt, from_root, src, n_src,
                                                   dst, n_dst, ev, n_ev, kb, cut, from_root ? a.window : 0, cnt);
        }
        if (meet) __syncwarp(live);
        if (!round_ok) {
            // a capacity was exceeded: redo this round from the root and stay in restart mode
            if (INSTR) cnt.fallbacks++;
            ckpt = false;
            from_root = true;
            n_ev = 0;
            kb.clear();
            trace_round<K, FORM, INSTR>(a, sc, o, d, inv, inv_len, tn, tf, Lt, Li, false, true, src, 0, dst, n_dst, ev, n_ev,
                                         kb, cut, 0, cnt);
        }
        for (int j = 0; j < kb.n; ++j) {
            uint32_t idx = kb.I(j) >> a.id_shift;
            blend_one<BWD>(a, sc, st, idx, o, d);
            if (INSTR) {
                if (a.ids && nb < a.ids_cap) a.ids[(size_t)pix * a.ids_cap + nb] = sc.gid[idx];
                cnt.blended++;
            }
            if (PASS == PASS_SAVE) save_blended(a, pix, nb, idx);
            ++nb;
            if (st.T < a.T_min) { done = true; break; }
        }
        first_round = false;
        if (done) continue;
        if (kb.n < K) {
            if (!(lim < GRTX_INF)) {
                done = true;
                continue;
            }
            // every hit up to the limit of the first round is blended: go on behind it, from the root
            Lt = lim;
            Li = GRTX_NONE;
            lim = GRTX_INF;
            cut.P = st.T;
            cut.far = 0.f;
            from_root = true;
            continue;
        }
        Lt = kb.T(K - 1);
        Li = kb.I(K - 1) >> a.id_shift;
        if (ckpt) {
            uint32_t tmp = src; src = dst; dst = tmp;
            n_src = n_dst;
            from_root = false;
        }
    }
    if (!BWD) out[pix] = make_float4(st.C[0] + st.T * a.bg0, st.C[1] + st.T * a.bg1, st.C[2] + st.T * a.bg2, st.T);
    if (INSTR && a.n_blended) a.n_blended[pix] = nb;
    if (PASS == PASS_SAVE) a.save_n[pix] = nb;
}

// The backward of a ray from the blend list its forward saved (n <= save_cap entries): the
// same blends, gradients and order as replaying the rounds, without the traversal.
__device__ __forceinline__ void backward_from_list(const TraceArgs &a, const SceneRef &sc, int64_t pix, float3 o,
                                                   float3 d, int n)
{
    BlendState st;
    st.C[0] = st.C[1] = st.C[2] = 0.f;
    st.T = 1.f;
    float4 F = a.fwd_rgbT[pix], G = a.dL_drgbT[pix];
    st.G[0] = G.x; st.G[1] = G.y; st.G[2] = G.z; st.G[3] = G.w;
    st.Tf = F.w;
    st.Cf[0] = F.x - F.w * a.bg0;
    st.Cf[1] = F.y - F.w * a.bg1;
    st.Cf[2] = F.z - F.w * a.bg2;
    st.dLdT = G.w + a.bg0 * G.x + a.bg1 * G.y + a.bg2 * G.z;
    const uint32_t *list = a.save_leaves + (size_t)pix * a.save_cap;
    for (int j = 0; j < n; ++j) {
        uint32_t idx = list[j];
        if (idx < sc.n_geom) blend_one<true>(a, sc, st, idx, o, d);   // never read outside the scene
    }
}

// The rays of one warp with restart traversal (Sec. III-A): every round from the root as the
// warp's packet over the lanes still tracing, each lane culling with its own last key L. Once
// rays travel as packets, the upper levels a restart revisits cost one broadcast load per warp,
// which is what makes this the faster restart on the SMs. A lane whose packet could not finish
// (the warp's stack would overflow) traces that round on its own. Every lane calls this
// together; lanes without a ray pass valid = false.
template <int K, int FORM, bool INSTR, bool SAVE>
__device__ __forceinline__ void trace_warp_restart(const TraceArgs &a, const SceneRef &sc, float4 *__restrict__ out,
                                                   int slot, bool valid, int64_t pix, float3 o, float3 d, float tn,
                                                   float tf, KBuf<K> &kb, Counters &cnt, uint4 *pst)
{
    if (!valid) {
        o = make_float3(0.f, 0.f, 0.f);
        d = make_float3(0.f, 0.f, 1.f);
        tn = tf = 0.f;
    }
    float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    float nrm = rsqrtf(d.x * d.x + d.y * d.y + d.z * d.z);
    BlendState st;
    st.C[0] = st.C[1] = st.C[2] = 0.f;
    st.T = 1.f;
    float Lt = tn;
    uint32_t Li = GRTX_NONE;
    int nb = 0;
    bool done = !valid || !sc.has_tree;
    Cut cut;                                   // unused: without an eviction list the k-buffer bounds a round
    cut.clear();
    while (__any_sync(0xffffffffu, !done)) {
        if (!done) {
            if (INSTR) cnt.rounds++;
            kb.clear();
        }
        int n_dst = 0, n_ev = 0;
        bool lane_ok = true;
        packet_round<K, FORM, INSTR>(a, sc, !done, pst, o, d, inv, nrm, tn, tf, Lt, Li, false, 0u, n_dst, 0u, n_ev,
                                     kb, cut, cnt, lane_ok);
        if (done) continue;
        if (!lane_ok) {
            kb.clear();
            trace_round<K, FORM, INSTR>(a, sc, o, d, inv, nrm, tn, tf, Lt, Li, false, true, 0u, 0, 0u, n_dst, 0u, n_ev,
                                        kb, cut, 0, cnt);
        }
        for (int j = 0; j < kb.n; ++j) {
            uint32_t idx = kb.I(j);
            blend_one<false>(a, sc, st, idx, o, d);
            if (INSTR) {
                if (a.ids && nb < a.ids_cap) a.ids[(size_t)pix * a.ids_cap + nb] = sc.gid[idx];
                cnt.blended++;
            }
            if (SAVE) save_blended(a, pix, nb, idx);
            ++nb;
            if (st.T < a.T_min) {
                done = true;
                break;
            }
        }
        if (!done && kb.n < K) done = true;
        if (!done) {
            Lt = kb.T(K - 1);
            Li = kb.I(K - 1);
        }
    }
    if (valid) {
        out[pix] = make_float4(st.C[0] + st.T * a.bg0, st.C[1] + st.T * a.bg1, st.C[2] + st.T * a.bg2, st.T);
        if (INSTR && a.n_blended) a.n_blended[pix] = nb;
        if (SAVE) a.save_n[pix] = nb;
    }
}

// The rays of one warp: round 1 as the warp's packet, then each ray's later rounds on its
// own. Every lane of the warp calls this together; lanes without a ray pass valid = false. In
// the backward, a ray whose forward saved its whole blend list takes it from there and leaves
// the traversal to the others.
template <int K, int FORM, bool INSTR, int PASS, bool WALK_ONLY = false, bool CHK = false, bool MEET = true>
__device__ __forceinline__ void trace_warp(const TraceArgs &a, const SceneRef &sc, float4 *__restrict__ out, int slot,
                                           bool valid, int64_t pix, float3 o, float3 d, float tn, float tf, KBuf<K> &kb,
                                           Counters &cnt, uint4 *pst)
{
    if (PASS == PASS_BWD && valid && a.save_n) {
        int n = a.save_n[pix];
        if (n <= a.save_cap) {
            backward_from_list(a, sc, pix, o, d, n);
            valid = false;
        }
    }
    if (!valid) {
        o = make_float3(0.f, 0.f, 0.f);
        d = make_float3(0.f, 0.f, 1.f);
        tn = tf = 0.f;
    }
    float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    float inv_len = rsqrtf(d.x * d.x + d.y * d.y + d.z * d.z);
    kb.clear();
    Cut cut;
    cut.clear();
    int n_dst = 0, n_ev = 0;
    bool lane_ok = true;
    float lim = GRTX_INF;
    constexpr bool WALKS = FORM == FORM_SPHERE && !INSTR;        // (where the lists are used)
    const bool walked = WALK_ONLY || (WALKS && a.traversal == GRTX_TRAVERSAL_CHECKPOINT);
    static_assert(sizeof(WalkShared) <= kWarpShared * sizeof(uint4), "the walk's shared memory");
    if (walked) {
        if (sc.has_tree && !tile_walk<K, CHK>(a, sc, valid, *reinterpret_cast<WalkShared *>(pst), o, d, tn, tf,
                                         a.ev_off + (uint32_t)slot, n_ev, kb, cut, lim, lane_ok)) {
            // a bundle that cannot be walked: its rays trace the round on their own, one to a warp where
            // the left list has room, or here
            // (kLeftRoom: more than the warps that can add to it after this check)
            if (PASS == PASS_FWD && a.left &&
                __all_sync(0xffffffffu, *reinterpret_cast<volatile unsigned *>(a.queue + 4) < kLeftCap - kLeftRoom)) {
                if ((threadIdx.x & 31) == 0) {
                    reinterpret_cast<WalkShared *>(pst)->rows = -1;
                    const unsigned to = atomicAdd(a.queue + 4, 1u);
                    if (in_bounds<CHK>(a, to, kLeftCap)) a.left[to] = reinterpret_cast<WalkShared *>(pst)->place;
                }
                return;
            }
            lane_ok = false;
        }
        const int most = __reduce_max_sync(0xffffffffu, valid && (!lane_ok || lim < GRTX_INF) ? 1 << 20 : n_ev);
        if ((threadIdx.x & 31) == 0)
            reinterpret_cast<WalkShared *>(pst)->rows = most >= (1 << 20) ? -1 : min(most, kDiscardRows);
        __syncwarp();
    } else {
        packet_round<K, FORM, INSTR>(a, sc, valid, pst, o, d, inv, inv_len, tn, tf, tn, GRTX_NONE,
                                     a.traversal == GRTX_TRAVERSAL_CHECKPOINT, a.ck1_off + (uint32_t)slot, n_dst,
                                     a.ev_off + (uint32_t)slot, n_ev, kb, cut, cnt, lane_ok);
    }
    // a lane whose packet could not finish (lists or the warp's stack overflowed) redoes round 1
    // from the root on its own, as after any capacity overflow. (Tried with its lists again first,
    // 1920x1080 of 6M 4-wide nodes took 27.1 instead of 17.1 ms.) One whose walk could not finish
    // begins anew: its bundle may only have shared too little.
    if (walked && !lane_ok) {
        cut.clear();
        lim = GRTX_INF;
    }
    const unsigned rays = __ballot_sync(0xffffffffu, valid);
    if (valid)
        trace_ray<K, FORM, INSTR, PASS, MEET>(a, sc, out, slot, pix, o, d, tn, tf, kb, cnt, cut, rays, !WALKS || lane_ok, WALKS || lane_ok,
                                        n_dst, n_ev, lim);
}

// After a tile, every checkpoint and eviction list entry of the warp's 32 ray slots is dead:
// the next tile writes each entry before it reads it. The lines holding them are dropped from
// L2 without being written back, so that the lists, written and read once per round, cost no
// DRAM writes. An entry row of the warp's slots is 32 x 8 = 256 contiguous bytes, two 128-byte
// lines, aligned because slot counts are multiples of 128 and list bases are 256-byte aligned.
// The first kDiscardRows rows of each list are dropped (a ray rarely writes more entries per
// round; a row past that is only written back as before); rows past a list's capacity would
// belong to the next list or lie past the workspace, and are skipped.

// After a walk only the eviction lists hold entries (rows: the longest list left, at most
// kDiscardRows; a list that was longer before it was shortened is seldom): 16 rows at a time.
__device__ __forceinline__ void discard_dead_lists(const TraceArgs &a, int warp_slot0, int rows)
{
    const size_t S = (size_t)a.n_slots;
    const int lane = threadIdx.x & 31;
    if (rows >= 0) {
        for (int r0 = 0; r0 < rows; r0 += 16) {
            const int row = r0 + (lane >> 1);
            if (row < rows) {
                const char *p = reinterpret_cast<const char *>(a.ev + (size_t)row * S + warp_slot0) + 128 * (lane & 1);
                asm volatile("discard.global.L2 [%0], 128;" ::"l"(p) : "memory");
            }
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < (3 * kDiscardRows * 2) / 32; ++q) {
        const int l = q * 32 + lane;
        const int list = l / (2 * kDiscardRows), row = (l % (2 * kDiscardRows)) >> 1, half = l & 1;
        const uint2 *base = list == 0 ? a.ck0 : (list == 1 ? a.ck1 : a.ev);
        const int cap = list == 2 ? a.evict_cap : a.ckpt_cap;
        if (row < cap) {
            const char *p = reinterpret_cast<const char *>(base + (size_t)row * S + warp_slot0) + 128 * half;
            asm volatile("discard.global.L2 [%0], 128;" ::"l"(p) : "memory");
        }
    }
}

// Resident blocks per SM the trace kernels are compiled for. The traversal is latency-bound,
// so occupancy pays even at the cost of a few spilled registers (measured on GB300: 8 blocks of
// 128 threads is the best forward setting for k <= 16; at k = 32 the k-buffer's 32 KB of shared memory
// allow 6 blocks, and 5 with a walk's 7.4 KB beside it; the backward keeps more live state and
// prefers 7).
__host__ __device__ constexpr int trace_min_blocks(int k, bool bwd) { return k >= 32 ? 6 : (bwd ? 7 : 8); }

// The item that queue place `place` of an image stands for: rows of tiles are handed out from the
// middle of the image outwards. A launch of more tiles than warps ends with its slowest tiles, and
// those lie where the scene is dense and deep, mostly around the middle (the horizon of an outdoor
// frame): started first, they run beside the others instead of after them. 6M outdoor frame and its
// bounce rays, 1920x1080, one launch: 11.7 -> 11.4 ms.
__device__ __forceinline__ unsigned middle_out(const CamRef &c, unsigned place)
{
    if (c.tiles_x == 0) return place;
    const unsigned tile = place >> 5, row = tile / (unsigned)c.tiles_x, mid = (unsigned)((c.height + 3) >> 2) >> 1;
    const unsigned to = (row & 1u) ? mid - ((row + 1u) >> 1) : mid + (row >> 1);
    return ((tile + (to - row) * (unsigned)c.tiles_x) << 5) | (place & 31u);
}

// Item of lane `lane` of the part of a tile that starts at queue place base: an 8x4 tile is taken
// in parts of 4x4, 4x2 or 2x2 pixels.
__device__ __forceinline__ unsigned split_item(const TraceArgs &a, unsigned base, int lane)
{
    if (a.middle) base = middle_out(a.cam, base);
    if (a.split == 0 || a.cam.tiles_x == 0) return base + (unsigned)lane;
    const unsigned part = (base & 31u) >> (5 - a.split), l = (unsigned)lane;
    const unsigned wx = a.split == 3 ? 1u : 2u;                              // log2 of a part's width
    const unsigned px = 3u - wx, x = ((part & ((1u << px) - 1u)) << wx) + (l & ((1u << wx) - 1u));
    const unsigned hy = a.split == 1 ? 2u : 1u;                              // log2 of a part's height
    const unsigned y = ((part >> px) << hy) + (l >> wx);
    return (base & ~31u) + y * 8u + x;
}

// How finely a launch of `tiles` 32-ray tiles is split over `warps` resident warps: halves, quarters
// or eighths of a tile while there are warps for them, since a tile's time is one warp's serial work.
// (256x256 preview 716 -> 553 us, 64x64 56 -> 45 us; the last part of the range, 1.25 tiles a warp,
// still gains: the parts differ more in time than a quarter.)
inline int split_for(unsigned tiles, unsigned warps, int most = 3)
{
    int s = 0;
    while (s < most && ((uint64_t)tiles << (s + 1)) <= (uint64_t)warps + warps / 4) ++s;
    return s;
}

// Traversal a frame kernel is compiled for: either (chosen per launch by a.traversal), or one
// of them only. The forward sphere-form kernel has one instantiation per traversal, and the
// checkpointed one none of the packet's code: without what does not run, the register allocation of
// what does is better (1M 1080p frame 3.591 -> 3.587 ms without the packet, a burst of 16 server requests
// 7.22 -> 7.16 ms).
// TRAV_CHECK: TRAV_CKPT with checked walks.
constexpr int TRAV_ANY = 0, TRAV_CKPT = 1, TRAV_RESTART = 2, TRAV_CHECK = 3;

template <int K, int FORM, bool INSTR, int PASS, int TRAV = TRAV_ANY>
__global__ void __launch_bounds__(kBlock, trace_min_blocks(K, PASS == PASS_BWD)) k_trace(TraceArgs a)
{
    __shared__ uint64_t s_k[K * kBlock];
    // the walk's shared memory or the packet's stack (with 3 KB instead of 7.6 a block, one more block
    // of a k = 32 restart launch fits)
    constexpr bool walks = FORM == FORM_SPHERE && !INSTR && TRAV != TRAV_RESTART;
    __shared__ uint4 s_pst[kBlock / 32][walks ? kWarpShared : kPacketStack];
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    KBuf<K> kb;
    kb.k = s_k + threadIdx.x;
    Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0, 0, nullptr, 0, 0};
    unsigned rays = 0;
    for (;;) {
        unsigned base = 0;
        const int take = walks ? 32 >> a.split : 32;
        if (lane == 0) base = atomicAdd(a.queue, (unsigned)take);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= a.n_items) break;
        int64_t pix;
        float3 o, d;
        float tn, tf;
        // (the kernels without a walk take whole tiles, and do without this arithmetic)
        bool valid = walks ? lane < take && make_ray(a.cam, split_item(a, base, lane), pix, o, d, tn, tf)
                           : make_ray(a.cam, base + lane, pix, o, d, tn, tf);
        if (walks && PASS == PASS_FWD && lane == 0) reinterpret_cast<WalkShared *>(s_pst[threadIdx.x >> 5])->place = make_uint2(base, 0u);
        rays += valid;
        if (INSTR) visits_begin(a, cnt, valid, pix);
        if constexpr (TRAV == TRAV_RESTART && PASS != PASS_BWD)
            trace_warp_restart<K, FORM, INSTR, PASS == PASS_SAVE>(a, a.sc, a.rgbT, slot, valid, pix, o, d, tn, tf,
                                                                  kb, cnt, s_pst[threadIdx.x >> 5]);
        else if constexpr (TRAV == TRAV_CKPT || TRAV == TRAV_CHECK)
            trace_warp<K, FORM, INSTR, PASS, true, TRAV == TRAV_CHECK, false>(a, a.sc, a.rgbT, slot, valid, pix, o, d, tn, tf, kb, cnt,
                                             s_pst[threadIdx.x >> 5]);
        else if (PASS != PASS_BWD && a.traversal == GRTX_TRAVERSAL_RESTART)
            trace_warp_restart<K, FORM, INSTR, PASS == PASS_SAVE>(a, a.sc, a.rgbT, slot, valid, pix, o, d, tn, tf,
                                                                  kb, cnt, s_pst[threadIdx.x >> 5]);
        else
            trace_warp<K, FORM, INSTR, PASS>(a, a.sc, a.rgbT, slot, valid, pix, o, d, tn, tf, kb, cnt,
                                             s_pst[threadIdx.x >> 5]);
        if (INSTR) visits_end(a, cnt, pix);
        __syncwarp();
        if (a.discard) {
            discard_dead_lists(a, slot & ~31, walks ? reinterpret_cast<WalkShared *>(s_pst[threadIdx.x >> 5])->rows : -1);
        }
    }
    if (INSTR && a.stats) {
        unsigned long long v[11] = {rays, cnt.nodes, cnt.leaves, cnt.blended, cnt.rounds, cnt.ckpt, cnt.evictions,
                                    cnt.fallbacks, cnt.overflow, 0ull, cnt.oob};
#pragma unroll
        for (int q = 0; q < 11; ++q) {
            unsigned long long x = v[q];
            for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
            if (lane == 0 && x) atomicAdd((&a.stats->rays) + q, x);
        }
    }
}

// The walk of one ray: every lane holds it, the lanes expand its pending nodes and take its leaves
// through the exact test side by side, and lane 0 collects the hits (its k-buffer and eviction list).
// False if the stack or the eviction list is too small.
template <int K, bool CHK = false>
__device__ __forceinline__ bool ray_walk(const TraceArgs &a, const SceneRef &sc, WalkShared &w, float3 o, float3 d, float tn,
                                         float tf, uint32_t ev, int &n_ev, KBuf<K> &kb, Cut &cut, float &lim)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t S = (uint32_t)a.n_slots;
    uint2 *const L = a.ck0;
    const float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    kb.clear();
    cut.clear();
    lim = GRTX_INF;
    n_ev = 0;
    float bound = tf;
    int squeeze_at = min(kSqueeze, max(a.evict_cap - 31, 1));
    bool ok = true;
    const int cap = a.packet_stack * (kWalkStack / kPacketStack), wide = cap - cap / 4;
    int sp = 1, nl = 0;
    __syncwarp();
    if (lane == 0) w.stack[0] = 0u;
    __syncwarp();
    for (;;) {
        if (sp >= cap || !__all_sync(full, ok)) return false;        // no room for children or hits
        const int p = min(min(32, sp), max(1, wide - sp));
        uint32_t cn = GRTX_NONE, cf = GRTX_NONE;
        if (lane < p && next_node<CHK>(a, sc, w, sp - 1 - lane)) {
            const float4 *nd = sc.nodes + 4 * (size_t)w.stack[sp - 1 - lane];
            const float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
            float e0, x0, e1, x1;
            slab(n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, o, inv, tn, bound, e0, x0);
            slab(n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, o, inv, tn, bound, e1, x1);
            cn = e0 <= x0 ? __float_as_uint(n3.x) : GRTX_NONE;
            cf = e1 <= x1 ? __float_as_uint(n3.y) : GRTX_NONE;
            if (e1 < e0) {
                const uint32_t t = cn; cn = cf; cf = t;
            }
            if (CHK) drop_bad_leaves(a, sc, cn, cf);
        }
        __syncwarp();
        const bool ln = cn != GRTX_NONE && (cn & GRTX_LEAF), lf = cf != GRTX_NONE && (cf & GRTX_LEAF);
        const unsigned bn = __ballot_sync(full, cn != GRTX_NONE && !ln), bf = __ballot_sync(full, cf != GRTX_NONE && !lf);
        const unsigned gn = __ballot_sync(full, ln), gf = __ballot_sync(full, lf);
        const unsigned below = (1u << lane) - 1u, above = ~(below | (1u << lane));
        sp -= p;
        int at = sp + __popc(bn & above) + __popc(bf & above);
        if (cf != GRTX_NONE && !lf && in_bounds<CHK>(a, at, kWalkStack)) w.stack[at++] = cf;
        if (cn != GRTX_NONE && !ln && in_bounds<CHK>(a, at, kWalkStack)) w.stack[at] = cn;
        sp += __popc(bn) + __popc(bf);
        at = nl + __popc(gn & below) + __popc(gf & below);
        if (ln && in_bounds<CHK>(a, at, kWalkLeaves)) w.leaf[at++] = cn & ~GRTX_LEAF;
        if (lf && in_bounds<CHK>(a, at, kWalkLeaves)) w.leaf[at] = cf & ~GRTX_LEAF;
        nl += __popc(gn) + __popc(gf);
        __syncwarp();
        if (sp > 0 && nl < 32) continue;
        for (int g0 = 0; g0 < nl; g0 += 32) {
            const int m = min(32, nl - g0);
            const uint32_t gi = w.leaf[g0 + min(lane, m - 1)];
            const float4 *g = sc.geom + 4 * (size_t)gi;
            const float4 r0 = __ldg(g), r1 = __ldg(g + 1), r2 = __ldg(g + 2), r3 = __ldg(g + 3);
            float t = 0.f, D2 = 0.f, q = 0.f, u[3], aa;
            bool hit = lane < m && sphere_candidate(r0, r1, r2, o, d, t, aa) && in_range(t, aa, tn, bound);
            if (hit) {
                sphere_refine(r0, r1, r2, o, d, t, D2, u);
                t = __fadd_rn(t, 0.0f);                              // (see sphere_test)
                hit = D2 <= 1.0f && t > tn && t <= tf && !(t > bound);
                q = 1.0f - fminf(r3.x * exp2f(r3.y * D2), a.alpha_max);
            }
            for (unsigned hits = __ballot_sync(full, hit); hits; hits &= hits - 1u) {
                const int h = __ffs(hits) - 1;
                float ct = __shfl_sync(full, t, h);
                const float hq = __shfl_sync(full, q, h);
                uint32_t ci = __shfl_sync(full, gi, h);
                if (lane == 0 && ok && !(ct > fminf(lim, cut.top(a)))) {
                    ci = cut.take(a, hq, ci, ct);
                    if (kb.insert(ct, ci)) {
                        if (n_ev >= a.evict_cap) {
                            ok = false;
                        } else {
                            if (in_bounds<CHK>(a, n_ev, a.evict_cap)) L[ev + (uint32_t)n_ev * S] = make_uint2(__float_as_uint(ct), ci);
                            ++n_ev;
                        }
                    }
                }
            }
            if (n_ev >= squeeze_at && ok) {                          // (its own lane only: the others have no hits)
                const bool no_room = n_ev + 32 > a.evict_cap;
                bool end;
                const float to = squeeze<K>(L + ev, S, n_ev, n_ev, kb.k,
                                            a.id_shift && a.p_stop > 0.f ? -__log2f(a.p_stop) : GRTX_INF, no_room, end);
                if (end) {
                    cut.P = 0.f;
                    cut.far = to;
                } else if (no_room) {
                    lim = to;
                }
                squeeze_at = min(n_ev + kSqueeze, max(a.evict_cap - 31, 1));
            }
            __syncwarp();
            bound = __shfl_sync(full, fminf(fminf(tf, lim), cut.top(a)), 0);
        }
        nl = 0;
        if (sp == 0) return __all_sync(full, ok);
    }
}

// The rays of the bundles that k_trace left (rays that share nothing, as scattered secondary rays do),
// one to a warp. Such a bundle traced per ray in k_trace is 32 lanes on 32 paths, about 500 steps that
// wait for memory one after another (and 626 warps are all that 20,011 rays give); here a ray is
// about 30 steps of up to 32 nodes, and every resident warp has one: 20,011 scattered rays over 1M
// Gaussians, k = 32, 1.90 -> 0.53 ms. The blend spreads over the lanes too: lane j takes entry j of the
// sorted k-buffer to its alpha and colour, then every lane composites them in order.
template <int K, bool CHK>
__global__ void __launch_bounds__(kBlock, 5) k_trace_rays(const __grid_constant__ TraceArgs a, const ServeSeg *segs)
{
    const unsigned full = 0xffffffffu;
    __shared__ uint64_t s_k[K * kBlock];
    __shared__ WalkShared s_w[kBlock / 32];
    const int slot = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const uint32_t ev = a.ev_off + (uint32_t)slot;
    const int take = 32 >> a.split;
    const unsigned n_left = min(a.queue[4], kLeftCap);
    KBuf<K> kb;
    kb.k = s_k + threadIdx.x;
    const uint64_t *keys = s_k + (threadIdx.x & ~31);            // lane 0's
    Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0, 0, nullptr, 0, 0};
    for (;;) {
        unsigned i = 0;
        if (lane == 0) i = atomicAdd(a.queue + 5, 1u);
        i = __shfl_sync(full, i, 0);
        if (i / (unsigned)take >= n_left) break;
        int64_t pix;
        float3 o, d;
        float tn, tf;
        const uint2 at = a.left[i / (unsigned)take];
        if (!segs && !in_bounds<CHK>(a, at.x, a.n_items)) continue;
        const int r = (int)(i % (unsigned)take);
        if (!(segs ? r < (32 >> segs[at.y].split) && make_ray(segs[at.y].cam, at.x + (unsigned)r, pix, o, d, tn, tf)
                   : make_ray(a.cam, split_item(a, at.x, r), pix, o, d, tn, tf)))
            continue;
        const SceneRef sc = segs ? segs[at.y].sc : a.sc;
        float4 *const out = segs ? segs[at.y].out : a.rgbT;
        Cut cut;
        float lim;
        int n_ev;
        const bool ok = ray_walk<K, CHK>(a, sc, s_w[threadIdx.x >> 5], o, d, tn, tf, ev, n_ev, kb, cut, lim);
        if (!ok || __shfl_sync(full, lim, 0) < GRTX_INF) {
            if (!ok) {                                           // it begins anew
                cut.clear();
                lim = GRTX_INF;
            }
            if (lane == 0)
                trace_ray<K, FORM_SPHERE, false, PASS_FWD>(a, sc, out, slot, pix, o, d, tn, tf, kb, cnt, cut, 1u, ok, true, 0,
                                                           n_ev, lim);
            __syncwarp();
            continue;
        }
        float C[3] = {0.f, 0.f, 0.f}, T = 1.f;
        for (;;) {
            const int n = __shfl_sync(full, kb.n, 0);
            float al = 0.f;
            float c[3] = {0.f, 0.f, 0.f};
            if (lane < n) al = blend_terms(a, sc, (uint32_t)keys[lane * kBlock] >> a.id_shift, o, d, c);
            bool done = false;
            for (int j = 0; j < n && !done; ++j) {
                const float aj = __shfl_sync(full, al, j), w = T * aj;
                C[0] = fmaf(w, __shfl_sync(full, c[0], j), C[0]);
                C[1] = fmaf(w, __shfl_sync(full, c[1], j), C[1]);
                C[2] = fmaf(w, __shfl_sync(full, c[2], j), C[2]);
                T *= 1.0f - aj;
                done = T < a.T_min;
            }
            if (done || n < K) break;
            __syncwarp();
            if (lane == 0) {                                      // the next K hits from the eviction list
                kb.clear();
                int k = 0;
                for (int e = 0; e < n_ev; ++e) {
                    uint2 v = a.ck0[ev + (uint32_t)e * (uint32_t)a.n_slots];
                    float ct = __uint_as_float(v.x);
                    uint32_t ci = v.y;
                    if (kb.insert(ct, ci)) {
                        a.ck0[ev + (uint32_t)k * (uint32_t)a.n_slots] = make_uint2(__float_as_uint(ct), ci);
                        ++k;
                    }
                }
                n_ev = k;
            }
            __syncwarp();
        }
        if (lane == 0) out[pix] = make_float4(C[0] + T * a.bg0, C[1] + T * a.bg1, C[2] + T * a.bg2, T);
        __syncwarp();
    }
}

// Acquire load (of a count the host raises after writing what it covers).
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr unsigned kLingerChecks = 1u << 16;   // bound on the checks of one wait (at most 8 us apart)

// Lane 0 of a warp of a serving launch that holds the claim `base`: returns base once the
// host has published the tile, or kNoWork when the launch is closed with base past its last
// item, or when linger_ns pass without any publication (each one restarts the wait). A warp
// that gives up puts its claim on the lost list (the host may publish it yet) and counts
// itself as exited. A warp about to wait writes its claim's end to claimed_host, so that the
// host sees the launch has run out of work.
__device__ __forceinline__ unsigned await_published(const ServeLive &live, unsigned base)
{
    const unsigned kNoWork = 0xffffffffu;
    unsigned seen = ld_acquire(live.avail);
    if (base < seen) return base;
    *reinterpret_cast<volatile unsigned *>(live.claimed_host) = base + 32u;
    uint64_t t0 = global_ns();
    unsigned nap = 64;
    for (unsigned it = 0; it < kLingerChecks; ++it) {
        const unsigned closed = ld_acquire(live.avail + 1);
        const unsigned n = ld_acquire(live.avail);
        if (base < n) return base;
        if (closed) return kNoWork;
        const uint64_t now = global_ns();
        if (n != seen) {
            seen = n;
            t0 = now;
        } else if (now - t0 > live.linger_ns) {
            break;
        }
        __nanosleep(nap);
        nap = min(2 * nap, 8192u);
    }
    const unsigned i = atomicAdd(live.lost, 1u);
    if (i < live.lost_cap) live.lost[1 + i] = base;
    const unsigned e = atomicAdd(live.exited, 1u) + 1u;
    *reinterpret_cast<volatile unsigned *>(live.exited_host) = e;
    return kNoWork;
}

// Serving step: one persistent launch over the queue items of several requests (each with
// its own scene, camera and output); a warp's 32 items always belong to one request.
template <int K, int TRAV>
__global__ void __launch_bounds__(kBlock, trace_min_blocks(K, false))
    k_serve(TraceArgs a, const ServeSeg *segs, const unsigned *begins, int n_segs, ServeLive live)
{
    __shared__ uint64_t s_k[K * kBlock];
    constexpr bool walks = TRAV == TRAV_CKPT;
    __shared__ uint4 s_pst[kBlock / 32][walks ? kWarpShared : kPacketStack];
    const unsigned kNoWork = 0xffffffffu;
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    KBuf<K> kb;
    kb.k = s_k + threadIdx.x;
    Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0, 0, nullptr, 0, 0};
    for (;;) {
        unsigned base = 0;
        if (lane == 0) {
            base = atomicAdd(a.queue, 32u);
            if (live.avail) {
                if ((base & 511u) == 0) *reinterpret_cast<volatile unsigned *>(live.claimed_host) = base + 32u;
                base = await_published(live, base);
            } else if (base >= a.n_items) {
                base = kNoWork;
            }
        }
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base == kNoWork) break;
        // last segment with begins[] <= base (read past L1: the host appends entries while the
        // launch runs; the entries not yet written hold 0xffffffff)
        int lo = 0, hi = n_segs - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (__ldcg(begins + mid) <= base) lo = mid; else hi = mid - 1;
        }
        // (a record is read only once its items are published, and fills whole cache lines of
        // its own, so no cache holds an older copy of it)
        const ServeSeg &sg = segs[lo];
        SceneRef sc = sg.sc;
        CamRef cam = sg.cam;
        unsigned item = sg.item_begin + (base - sg.step_begin);
        if (a.middle) item = middle_out(cam, item);
        const int take = 32 >> sg.split;
        item = (item >> sg.split) + (unsigned)lane;
        int64_t pix;
        float3 o, d;
        float tn, tf;
        bool valid = lane < take && make_ray(cam, item, pix, o, d, tn, tf);
        if (walks && a.left && lane == 0)
            reinterpret_cast<WalkShared *>(s_pst[threadIdx.x >> 5])->place = make_uint2(item, (unsigned)lo);
        if constexpr (TRAV == TRAV_RESTART)
            trace_warp_restart<K, FORM_SPHERE, false, false>(a, sc, sg.out, slot, valid, pix, o, d, tn, tf, kb, cnt,
                                                      s_pst[threadIdx.x >> 5]);
        else
            trace_warp<K, FORM_SPHERE, false, PASS_FWD, true>(a, sc, sg.out, slot, valid, pix, o, d, tn, tf, kb, cnt,
                                                     s_pst[threadIdx.x >> 5]);
        if (live.seg_done) {
            // the tile's pixels are written; the warp that completes the segment raises its
            // flag in host memory (each lane's writes fenced before the count)
            __threadfence();
            __syncwarp();
            if (lane == 0) {
                const unsigned old = atomicAdd(live.seg_done + lo, 32u);
                if (old + 32u >= sg.count) {
                    __threadfence_system();
                    *reinterpret_cast<volatile unsigned *>(live.seg_flag + lo) = live.seq;
                }
            }
        }
        __syncwarp();
        if (a.discard) {
            discard_dead_lists(a, slot & ~31, walks ? reinterpret_cast<WalkShared *>(s_pst[threadIdx.x >> 5])->rows : -1);
        }
    }
}

// Entry offsets of the lists relative to ck0 (the kernels index every list entry with 32 bits);
// false if the workspace is too large for that. Call after ck0, ck1, ev and n_slots are set.
inline bool set_list_offsets(TraceArgs &a, size_t entries_per_slot)
{
    if ((size_t)a.n_slots * entries_per_slot >= ((size_t)1 << 31)) return false;
    a.ck1_off = (uint32_t)(a.ck1 - a.ck0);
    a.ev_off = (uint32_t)(a.ev - a.ck0);
    return true;
}

// The first round's window and the opacity at which a ray is known to end (see Cut). The window
// leaves room in both lists: with the default capacities (256 / 512) it is 64 hits.
inline void set_window(TraceArgs &a)
{
    const int cap = a.ckpt_cap < a.evict_cap ? a.ckpt_cap : a.evict_cap;
    a.window = a.traversal == GRTX_TRAVERSAL_CHECKPOINT ? cap / 4 : 0;
    a.p_stop = a.T_min >= 1e-30f ? 0.98f * a.T_min : 0.0f;
    a.id_shift = 0;
    a.leave_at = 0x7fffffff;
}

// Opacity codes in the list entries: for the walk (uninstrumented sphere-form kernels), where the
// largest scene's leaf slots leave room for them.
inline void set_codes(TraceArgs &a, int form, bool instr, int64_t n_valid)
{
    const bool walk = form == FORM_SPHERE && !instr && a.traversal == GRTX_TRAVERSAL_CHECKPOINT;
    a.id_shift = walk && n_valid < ((int64_t)1 << (32 - kCodeBits)) ? kCodeBits : 0;
}

// Whether the lists of a launch may be dropped from L2 per tile (see discard_dead_lists): the
// checkpointed traversal writes lists, and each list row must start on a 256-byte boundary.
inline int lists_discardable(const TraceArgs &a)
{
    if (a.traversal != GRTX_TRAVERSAL_CHECKPOINT || !a.ck0 || !a.ck1 || !a.ev) return 0;
    const uintptr_t m = (uintptr_t)a.ck0 | (uintptr_t)a.ck1 | (uintptr_t)a.ev;
    return (m & 255u) == 0 && (a.n_slots % 32) == 0 && ((size_t)a.n_slots * sizeof(uint2)) % 256 == 0;
}

// k of the checked kernels (the walks are the same for every k).
constexpr int kCheckK = 16;

// Launch helpers, instantiated per k in the trace_k*.cu units.
// form: FORM_* of the scene. The backward always runs the sphere leaf test: the icosphere
// forms hit exactly the Gaussians the sphere form hits, and the proxy form has no backward.
// pass: PASS_FWD, PASS_BWD or PASS_SAVE (the saving forward exists for the sphere form only).
template <int K>
int trace_launch(const TraceArgs &a, int form, bool instr, int pass, int blocks, cudaStream_t s)
{
    dim3 g(blocks), b(128);
    if (pass == PASS_BWD) k_trace<K, FORM_SPHERE, false, PASS_BWD><<<g, b, 0, s>>>(a);
    else if (pass == PASS_SAVE) k_trace<K, FORM_SPHERE, false, PASS_SAVE><<<g, b, 0, s>>>(a);
    else if (form == FORM_PROXY && instr) k_trace<K, FORM_PROXY, true, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (form == FORM_PROXY) k_trace<K, FORM_PROXY, false, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (form == FORM_ICO && instr) k_trace<K, FORM_ICO, true, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (form == FORM_ICO) k_trace<K, FORM_ICO, false, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (form == FORM_SPHERE4 && instr) k_trace<K, FORM_SPHERE4, true, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (form == FORM_SPHERE4) k_trace<K, FORM_SPHERE4, false, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (form == FORM_SPHERE4Q && instr) k_trace<K, FORM_SPHERE4Q, true, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (form == FORM_SPHERE4Q) k_trace<K, FORM_SPHERE4Q, false, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (instr) k_trace<K, FORM_SPHERE, true, PASS_FWD><<<g, b, 0, s>>>(a);
    else if (a.traversal == GRTX_TRAVERSAL_RESTART) k_trace<K, FORM_SPHERE, false, PASS_FWD, TRAV_RESTART><<<g, b, 0, s>>>(a);
    else if (K == kCheckK && a.check) k_trace<K, FORM_SPHERE, false, PASS_FWD, K == kCheckK ? TRAV_CHECK : TRAV_CKPT><<<g, b, 0, s>>>(a);
    else k_trace<K, FORM_SPHERE, false, PASS_FWD, TRAV_CKPT><<<g, b, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? GRTX_OK : GRTX_ERR_CUDA;
}

template <int K>
int trace_rays_launch(const TraceArgs &a, const ServeSeg *segs, int blocks, cudaStream_t s)
{
    if (K == kCheckK && a.check) k_trace_rays<K, K == kCheckK><<<blocks, kBlock, 0, s>>>(a, segs);
    else k_trace_rays<K, false><<<blocks, kBlock, 0, s>>>(a, segs);
    return cudaGetLastError() == cudaSuccess ? GRTX_OK : GRTX_ERR_CUDA;
}

// Blocks per multiprocessor of the kernel that trace_launch takes for the same arguments. (The restart
// kernel keeps no walk and fits 6 blocks at k = 32, the checkpointed one 5: sized by the latter, a
// restarted 1M 1080p frame took 9.0 instead of 8.1 ms.)
template <int K>
int trace_occupancy(int form, bool instr, int pass, int traversal, int *blocks_per_sm)
{
    cudaError_t e;
    if (pass == PASS_BWD) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE, false, PASS_BWD>, 128, 0);
    else if (pass == PASS_SAVE) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE, false, PASS_SAVE>, 128, 0);
    else if (form == FORM_PROXY && instr) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_PROXY, true, PASS_FWD>, 128, 0);
    else if (form == FORM_PROXY) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_PROXY, false, PASS_FWD>, 128, 0);
    else if (form == FORM_ICO && instr) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_ICO, true, PASS_FWD>, 128, 0);
    else if (form == FORM_ICO) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_ICO, false, PASS_FWD>, 128, 0);
    else if (form == FORM_SPHERE4 && instr) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE4, true, PASS_FWD>, 128, 0);
    else if (form == FORM_SPHERE4) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE4, false, PASS_FWD>, 128, 0);
    else if (form == FORM_SPHERE4Q && instr) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE4Q, true, PASS_FWD>, 128, 0);
    else if (form == FORM_SPHERE4Q) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE4Q, false, PASS_FWD>, 128, 0);
    else if (instr) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE, true, PASS_FWD>, 128, 0);
    else if (traversal == GRTX_TRAVERSAL_RESTART) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE, false, PASS_FWD, TRAV_RESTART>, 128, 0);
    else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_trace<K, FORM_SPHERE, false, PASS_FWD, TRAV_CKPT>, 128, 0);
    return e == cudaSuccess ? GRTX_OK : GRTX_ERR_CUDA;
}

// Kernel leaf kind of a scene form (wide: the 4-wide nodes of a sphere-form scene, quantised
// or not).
inline int kernel_form(int scene_form, bool wide = false, bool quant = false)
{
    return scene_form == GRTX_FORM_PROXY20 ? FORM_PROXY
           : (scene_form == GRTX_FORM_ICO20 || scene_form == GRTX_FORM_ICO80) ? FORM_ICO
           : wide ? (quant ? FORM_SPHERE4Q : FORM_SPHERE4) : FORM_SPHERE;
}

// live: the serving controls (see ServeLive); all zero for a plain batched launch.
template <int K>
int serve_launch(const TraceArgs &a, const ServeSeg *segs, const unsigned *begins, int n_segs, int blocks,
                 cudaStream_t s, ServeLive live)
{
    if (a.traversal == GRTX_TRAVERSAL_RESTART) k_serve<K, TRAV_RESTART><<<blocks, 128, 0, s>>>(a, segs, begins, n_segs, live);
    else k_serve<K, TRAV_CKPT><<<blocks, 128, 0, s>>>(a, segs, begins, n_segs, live);
    return cudaGetLastError() == cudaSuccess ? GRTX_OK : GRTX_ERR_CUDA;
}

template <int K>
int serve_occupancy(int traversal, int *blocks_per_sm)
{
    const cudaError_t e = traversal == GRTX_TRAVERSAL_RESTART
                              ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_serve<K, TRAV_RESTART>, 128, 0)
                              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_serve<K, TRAV_CKPT>, 128, 0);
    return e == cudaSuccess ? GRTX_OK : GRTX_ERR_CUDA;
}

#define GRTX_INSTANTIATE_TRACE(K)                                                                  \
    template int trace_launch<K>(const TraceArgs &, int, bool, int, int, cudaStream_t);           \
    template int trace_occupancy<K>(int, bool, int, int, int *);                                         \
    template int trace_rays_launch<K>(const TraceArgs &, const ServeSeg *, int, cudaStream_t);                        \
    template int serve_launch<K>(const TraceArgs &, const ServeSeg *, const unsigned *, int, int, cudaStream_t, ServeLive);   \
    template int serve_occupancy<K>(int, int *);
