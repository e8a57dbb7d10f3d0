// Primary-ray tracer: emission (Eq. 6), traversal with reflection/refraction
// at analytic boundaries (Eqs. 7-11), transducer sampling of point scatterers
// through straight connection rays with the receive directivity (Eq. 13), and
// recording of returns to the aperture.  FP32 geometry, float-float time of
// flight; arrivals are appended to a global queue for the binning stage.  The kernel template and
// its device code; the ur_trace*.cu files compile its instantiations in parallel.
#pragma once

#include "ur_device.cuh"

namespace ur {
namespace {

// Philox blocks of the plane-wave tracer come from one out-of-line copy: the kernel's hot loop
// stays smaller, and instruction fetch is its first stall (layered frame 8.59 -> 8.17 ms); the
// extended tracers keep them inline (there the call cost more than the code it saved).
__device__ __noinline__ uint4 philox_outline(uint4 c, uint2 k) { return philox(c, k); }

template <bool INLINE>
__device__ __forceinline__ uint4 draw(uint4 c, uint2 k) { return INLINE ? philox(c, k) : philox_outline(c, k); }

// Straight connection ray from p to the element centre (x_e, 0, 0): product of
// sqrt(1 - R) over the boundaries it crosses (0 if one reflects totally),
// travel time (samples) and attenuation exponent.  skip0: the boundary p lies
// on (-1 inside a medium).
template <bool MESH>
__device__ float connection(const SceneP &S, float3 p, int med, int skip0, float xe, ff &t_conn, float &att) {
    float3 o = p;
    float3 w = make_float3(xe - p.x, -p.y, -p.z);
    const float w2 = dot3_yx(w, w), iw = rsqrtf(w2);
    float rem = sqrtf(w2);   // the length sets the travel time: correctly rounded
    w = make_float3(w.x * iw, w.y * iw, w.z * iw);
    float fac = 1.f, a = 0.f;
    ff t = {0.f, 0.f};
    int m = med, skip = skip0;
    for (int it = 0; it < kMaxCross; ++it) {
        float th;
        const int hit = nearest<MESH, true>(S, o, w, skip, false, th);
        const Medium &M = S.med[m];
        if (hit < 0 || th >= rem) {
            t = ff_add(t, ff_mul_f(rem, M.slow));
            a = fmaf(M.a, rem, a);
            break;
        }
        t = ff_add(t, ff_mul_f(th, M.slow));
        a = fmaf(M.a, th, a);
        float3 h = along(o, th, w), n;
        int m_neg, m_pos;
        float alpha;
        surface<MESH>(S, hit, h, n, m_neg, m_pos, alpha);
        const float dn = dot3(w, n);
        const int m2 = dn > 0.f ? m_pos : m_neg;
        float r, ct;
        if (!fresnel(fabsf(dn), M.c, M.Z, S.med[m2].c, S.med[m2].Z, r, ct)) return 0.f;
        fac *= sqrtf(transmitted(fabsf(dn), ct, M.Z, S.med[m2].Z));
        m = m2;
        o = h;
        rem -= th;
        skip = hit;
    }
    t_conn = t;
    att = a;
    return fac;
}

// ---------------------------------------------------------------- rough boundaries (Eq. 12)
constexpr float kPiF = 3.14159265358979f;

// GGX density of microfacet normals at c = n.h, a2 = alpha^2; the denominator
// written as (1 - c^2) + a2 c^2 stays positive when c rounds to 1.
__device__ __forceinline__ float ggx_d(float c, float a2) {
    if (!(c > 0.f)) return 0.f;
    const float c2 = __fmul_rn(c, c);
    const float k = fmaf(a2, c2, __fsub_rn(1.f, c2));
    return a2 / (kPiF * k * k);
}

// Smith masking of one direction at cosine c to the macro normal.
__device__ __forceinline__ float ggx_g1(float c, float a2) {
    const float c2 = __fmul_rn(c, c);
    const float t2 = __fsub_rn(1.f, c2) / c2;
    return 2.f / (1.f + sqrtf(fmaf(a2, t2, 1.f)));
}

// Microfacet normal with density D(m)(m.n) about unit n: tan^2 theta = alpha^2 xi1 / (1 - xi1),
// phi = 2 pi xi2, in the tangent frame of Duff et al. (JCGT 2017).
__device__ __forceinline__ float3 ggx_sample(float3 n, float a2, float xi1, float xi2, float &ct) {
    const float tan2 = a2 * xi1 / (1.f - xi1);
    ct = 1.f / sqrtf(1.f + tan2);
    const float st = sqrtf(tan2) * ct;
    float sp, cp;
    sincospif(2.f * xi2, &sp, &cp);
    const float sg = n.z >= 0.f ? 1.f : -1.f;
    const float a = -1.f / (sg + n.z);
    const float b = n.x * n.y * a;
    const float3 t1 = make_float3(fmaf(__fmul_rn(__fmul_rn(sg, n.x), n.x), a, 1.f), sg * b, -sg * n.x);
    const float3 t2 = make_float3(b, fmaf(__fmul_rn(n.y, n.y), a, sg), -n.y);
    return along(blend(st * cp, t1, st * sp, t2), ct, n);
}

// Scattering of a rough boundary from incident direction d (n: unit macro normal
// on the incident side) into o: returns f |o.n| in the amplitude form (r or
// sqrt(1 - R) of the half-vector microfacet) and the solid-angle density of o
// under microfacet sampling and the reflect-if-y < R branch.
__device__ float rough_eval(float3 d, float3 n, float3 o, float a2, const Medium &M1, const Medium &M2,
                           float &pdf) {
    pdf = 0.f;
    const float3 i = make_float3(-d.x, -d.y, -d.z);
    const float cos_i = dot3_yx(i, n), cos_o = dot3_yx(o, n);
    if (!(cos_i > 0.f) || cos_o == 0.f) return 0.f;
    float3 h;
    float coef, pb, jac;
    if (cos_o > 0.f) {
        h = i + o;
        const float il = rsqrtf(dot3_yx(h, h));
        h = make_float3(h.x * il, h.y * il, h.z * il);
        const float ih = dot3(i, h);
        if (!(dot3(h, n) > 0.f) || !(ih > 0.f)) return 0.f;
        float r, ct;
        const bool ok = fresnel(ih, M1.c, M1.Z, M2.c, M2.Z, r, ct);
        coef = ok ? r : 1.f;
        pb = ok ? r * r : 1.f;
        jac = 0.25f / dot3(o, h);
    } else {
        const float eta = M2.c / M1.c;
        h = unit3(along(o, eta, i));   // along i/c1 + o/c2
        if (dot3(h, n) < 0.f) h = make_float3(-h.x, -h.y, -h.z);
        const float ih = dot3(i, h), oh = dot3(o, h);
        if (!(dot3(h, n) > 0.f) || !(ih > 0.f) || !(oh < 0.f)) return 0.f;
        float r, ct;
        if (!fresnel(ih, M1.c, M1.Z, M2.c, M2.Z, r, ct)) return 0.f;
        const float den = fmaf(eta, ih, oh);   // c2 (i.h / c1 + o.h / c2)
        if (!(den * den > 1e-30f)) return 0.f;
        pb = transmitted(ih, ct, M1.Z, M2.Z);
        coef = sqrtf(pb);
        jac = -oh / (den * den);
    }
    const float hn = dot3(h, n);
    const float D = ggx_d(hn, a2);
    const float G = ggx_g1(cos_i, a2) * ggx_g1(fabsf(cos_o), a2);
    pdf = D * hn * jac * pb;
    return coef * G * D * dot3_yx(i, h) * jac / cos_i;
}

// The same toward an arbitrary element centre q (convex arrays).
template <bool MESH>
__device__ float connection_to(const SceneP &S, float3 p, int med, int skip0, float3 q, ff &t_conn, float &att) {
    float3 o = p;
    float3 w = make_float3(q.x - p.x, q.y - p.y, q.z - p.z);
    const float w2 = dot3_yx(w, w), iw = rsqrtf(w2);
    float rem = sqrtf(w2);   // the length sets the travel time: correctly rounded
    w = make_float3(w.x * iw, w.y * iw, w.z * iw);
    float fac = 1.f, a = 0.f;
    ff t = {0.f, 0.f};
    int m = med, skip = skip0;
    for (int it = 0; it < kMaxCross; ++it) {
        float th;
        const int hit = nearest<MESH, false, true>(S, o, w, skip, false, th);
        const Medium &M = S.med[m];
        if (hit < 0 || th >= rem) {
            t = ff_add(t, ff_mul_f(rem, M.slow));
            a = fmaf(M.a, rem, a);
            break;
        }
        t = ff_add(t, ff_mul_f(th, M.slow));
        a = fmaf(M.a, th, a);
        float3 h = along(o, th, w), n;
        int m_neg, m_pos;
        float alpha;
        surface<MESH>(S, hit, h, n, m_neg, m_pos, alpha);
        const float dn = dot3(w, n);
        const int m2 = dn > 0.f ? m_pos : m_neg;
        float r, ct;
        if (!fresnel(fabsf(dn), M.c, M.Z, S.med[m2].c, S.med[m2].Z, r, ct)) return 0.f;
        fac *= sqrtf(transmitted(fabsf(dn), ct, M.Z, S.med[m2].Z));
        m = m2;
        o = h;
        rem -= th;
        skip = hit;
    }
    t_conn = t;
    att = a;
    return fac;
}

// Centre c and unit normal n of element e: on the arc of a convex array (radius > 0;
// z written as -2 R sin^2(phi/2) to avoid cancellation near the apex), else (x_e, 0, 0), +z.
template <bool CVX>
__device__ __forceinline__ void elem_frame(const TraceP &P, uint32_t e, float3 &c, float3 &n) {
    if (CVX) {
        const float ph = fmaf((float)e, P.dphi, P.phi0);
        float sn, cs, sh, ch;
        sincosf(ph, &sn, &cs);
        sincosf(0.5f * ph, &sh, &ch);
        n = make_float3(sn, 0.f, cs);
        c = make_float3(P.radius * sn, 0.f, -2.f * P.radius * sh * sh);
    } else {
        c = make_float3(fmaf((float)e, P.pitch, P.x_first), 0.f, 0.f);
        n = make_float3(0.f, 0.f, 1.f);
    }
}

// The scene of a lane: launches of one scene (every ur_trace) read its parameters as kernel constants
// instead of per-lane indexed loads (layered frame 5578 -> 4991 us).
template <int GEO>
__device__ __forceinline__ const SceneP &scene_of(const TraceP &P, int scene) {
    return (GEO & kGeoOne) ? P.S[0] : P.S[scene];
}

// Warp-aggregated append to the arrival queue (one atomic per converged group);
// with DBG or REC the arrival's (ray, event) words go to arr_dbg as well.
template <bool DBG, bool REC>
__device__ __forceinline__ void emit(const TraceP &P, uint32_t row, ff t, float amp, uint32_t ray, uint32_t ev) {
    const unsigned mask = __activemask();
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(mask) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(P.arr_count, (unsigned long long)__popc(mask));
    base = __shfl_sync(mask, base, leader);
    const unsigned long long idx = base + (unsigned long long)__popc(mask & ((1u << lane) - 1u));
    if (idx < P.arr_cap) {
        P.arr[idx] = make_uint4(row, __float_as_uint(t.hi), __float_as_uint(t.lo), __float_as_uint(amp));
        if (DBG || REC) P.arr_dbg[idx] = make_uint2(ray, ev);
    }
}

struct Counters {
    uint32_t rays, segments, interactions, candidates, connections, arrivals;
};

constexpr int kBlock = 256;
constexpr int kWarps = kBlock / 32;
constexpr int kQueue = 64;     // scatterer-event ring per warp (power of two, >= 63 entries needed)
constexpr int kPool = kTracePool;

// Lane states: a segment to be finished, waiting for a new ray, ray placed or redirected (its next
// segment to be set up), no rays left.
enum { kHasSeg = 0, kNeedRay = 1, kNeedSeg = 2, kFinished = 3 };

// Scatterer events waiting for their connection ray, one ring per warp (SoA).
struct WarpQueue {
    uint32_t ray[kQueue], kmb[kQueue], j[kQueue];
    float tca[kQueue], t_hi[kQueue], t_lo[kQueue], w[kQueue];
};

// A batch of column visits: the lanes whose segments have any, and the visits that hold references:
// (segment's lane | kWalkFine, first reference minus its number in the batch, t_enter, t_end).
struct WarpVisits {
    uint4 visit[32];
    uint32_t seg_lane[32];
};

// Column walk of a segment (Lane::walk): first column along its main axis, and
constexpr uint32_t kWalkY = 1u << 28;      // the main axis is y
constexpr uint32_t kWalkDual = 1u << 29;   // the other axis' column changes on the way
constexpr uint32_t kWalkNeg = 1u << 30;    // columns are passed downwards
constexpr uint32_t kWalkFine = 1u << 31;   // one visit of a fine column (vertical segments)
constexpr uint32_t kWalkCell = kWalkY - 1u;

// Per-lane state: the primary ray, its current segment and the stretch of it inside the grid box.
struct Lane {
    float3 o, d;
    ff t;
    float w, L;
    int med, b, prev, scene;
    uint32_t i, item, stream;
    uint64_t h;
    float seg;
    int hit;
    bool clipped;
    float t0, t1;
    uint32_t walk;
    int state;
    // rough boundaries: the path left a rough vertex mp with direction density mpdf and has
    // crossed only by transmission since (its aperture hit takes a balance-heuristic weight)
    bool mis;
    float3 mp;
    float mpdf;
};

__device__ __forceinline__ uint32_t lanemask_lt() { return (1u << (threadIdx.x & 31)) - 1u; }

__device__ __forceinline__ int cell_at(float x, float lo, float inv_h, int dim) {
    return min(max((int)floorf((x - lo) * inv_h), 0), dim - 1);
}

// Segment from the current position to the nearest boundary (clipped by the path-length budget),
// and the column visits of its part inside the grid box: returns their number.  The visits step
// along the axis on which the segment passes more columns; where the other axis' column changes on
// the way, each step is two visits, before and after that change (at most one per step, up to
// rounding that the references' margin g_rm absorbs).
template <int GEO, bool FINE>
__device__ __forceinline__ uint32_t start_segment(const TraceP &P, Lane &R, Counters &cn) {
    constexpr bool CVX = (GEO & kGeoConvex) != 0, MESH = (GEO & kGeoMesh) != 0;
    const SceneP &S = scene_of<GEO>(P, R.scene);
    float th;
    R.hit = nearest<MESH>(S, R.o, R.d, R.prev, true, th, CVX ? P.radius : 0.f);
    R.seg = th;
    R.clipped = false;
    if (R.L + R.seg > P.max_path) {
        R.seg = P.max_path - R.L;
        R.clipped = true;
    }
    cn.segments++;
    R.state = kHasSeg;
    if (S.n_scat == 0) return 0u;
    const float3 o = R.o, d = R.d;
    const float hi_x = S.g_lo.x + (float)S.g_dim.x * S.g_h.x;
    const float hi_y = S.g_lo.y + (float)S.g_dim.y * S.g_h.y;
    const float hi_z = S.g_lo.z + (float)S.g_dim.z * S.g_h.z;
    float t0 = 0.f, t1 = R.seg;
    // Reciprocals of the direction for the box clip and the column steps.  They only place
    // column boundaries, which the g_rm margin of the references absorbs, so the approximate
    // form serves (a few ulp, and no slow path for the zero components of in-plane and
    // vertical rays: in a y-invariant scene every ray has d.y = 0).
    const float ix = __fdividef(1.f, d.x), iy = __fdividef(1.f, d.y), iz = __fdividef(1.f, d.z);
    if (d.x != 0.f) {
        const float ta = (S.g_lo.x - o.x) * ix, tb = (hi_x - o.x) * ix;
        t0 = fmaxf(t0, fminf(ta, tb));
        t1 = fminf(t1, fmaxf(ta, tb));
    } else if (o.x < S.g_lo.x || o.x > hi_x) {
        return 0u;
    }
    if (d.y != 0.f) {
        const float ta = (S.g_lo.y - o.y) * iy, tb = (hi_y - o.y) * iy;
        t0 = fmaxf(t0, fminf(ta, tb));
        t1 = fminf(t1, fmaxf(ta, tb));
    } else if (o.y < S.g_lo.y || o.y > hi_y) {
        return 0u;
    }
    if (d.z != 0.f) {
        const float ta = (S.g_lo.z - o.z) * iz, tb = (hi_z - o.z) * iz;
        t0 = fmaxf(t0, fminf(ta, tb));
        t1 = fminf(t1, fmaxf(ta, tb));
    } else if (o.z < S.g_lo.z || o.z > hi_z) {
        return 0u;
    }
    if (!(t0 < t1)) return 0u;
    R.t0 = t0;
    R.t1 = t1;
    if (FINE && d.x == 0.f && d.y == 0.f && S.f_refs) {   // vertical: one visit of a fine column
        R.walk = kWalkFine;
        return 1u;
    }
    const int x0 = cell_at(o.x + t0 * d.x, S.g_lo.x, S.g_inv_h.x, S.g_dim.x);
    const int x1 = cell_at(o.x + t1 * d.x, S.g_lo.x, S.g_inv_h.x, S.g_dim.x);
    const int y0 = cell_at(o.y + t0 * d.y, S.g_lo.y, S.g_inv_h.y, S.g_dim.y);
    const int y1 = cell_at(o.y + t1 * d.y, S.g_lo.y, S.g_inv_h.y, S.g_dim.y);
    const bool along_y = fabsf(d.y) * S.g_inv_h.y > fabsf(d.x) * S.g_inv_h.x;
    const int c0 = along_y ? y0 : x0, c1 = along_y ? y1 : x1;
    const bool dual = along_y ? x0 != x1 : y0 != y1;
    const uint32_t n = (uint32_t)abs(c1 - c0) + 1u;
    R.walk = (uint32_t)c0 | (along_y ? kWalkY : 0u) | (dual ? kWalkDual : 0u) | (c1 < c0 ? kWalkNeg : 0u);
    return dual ? 2u * n : n;
}

// Visit k of the n of a segment o + t d (walk, box stretch [t0, t1], length seg): the references
// `begin` .. `begin` + count of one column's z cells within g_rm of the depths its stretch spans, and
// the stretch [t_enter, t_end) whose closest approaches it accepts.  The stretches of a segment's
// visits share their ends (the same expression gives both) and none but the last passes t1, so every
// scatterer within r_s of the segment is accepted exactly once; the first reaches g_rm before the
// box and the last to the segment's end (no closest approach lies outside the box, the margins only
// keep rounding out of play).
template <bool FINE>
__device__ __forceinline__ uint32_t column_visit(const SceneP &S, float3 o, float3 d, uint32_t walk, float t0, float t1,
                                                 float seg, uint32_t k, uint32_t n, uint32_t &begin,
                                                 float &t_enter, float &t_end) {
    float ta = t0, tb = t1;
    t_enter = t0 - S.g_rm;
    t_end = seg;
    const bool fine = FINE && (walk & kWalkFine);
    int cx, cy;
    if (fine) {
        cx = cell_at(o.x, S.f_lo.x, S.f_inv_h.x, S.f_dim.x);
        cy = cell_at(o.y, S.f_lo.y, S.f_inv_h.y, S.f_dim.y);
    } else {
        const bool dual = (walk & kWalkDual) != 0u, neg = (walk & kWalkNeg) != 0u, along_y = (walk & kWalkY) != 0u;
        const bool second = dual && (k & 1u);
        if (dual) {
            k >>= 1;
            n >>= 1;
        }
        const int c = (int)(walk & kWalkCell) + (neg ? -(int)k : (int)k);
        const float om = along_y ? o.y : o.x, os = along_y ? o.x : o.y;
        const float dm = along_y ? d.y : d.x, ds = along_y ? d.x : d.y;
        const float lom = along_y ? S.g_lo.y : S.g_lo.x, los = along_y ? S.g_lo.x : S.g_lo.y;
        const float hm = along_y ? S.g_h.y : S.g_h.x, hs = along_y ? S.g_h.x : S.g_h.y;
        const float inv_hs = along_y ? S.g_inv_h.x : S.g_inv_h.y;
        const int dim_s = along_y ? S.g_dim.x : S.g_dim.y;
        const float im = __fdividef(1.f, dm);
        const auto border = [&](int b) { return (fmaf((float)b, hm, lom) - om) * im; };   // column b's lower side
        if (k > 0u) t_enter = ta = border(neg ? c + 1 : c);
        // for a ray that hardly crosses the columns, im magnifies the rounding of the side past the end
        if (k + 1u < n) t_end = tb = fminf(border(neg ? c : c + 1), t1);
        const int sa = cell_at(os + ta * ds, los, inv_hs, dim_s);
        int cs = sa;
        if (dual) {
            const int sb = cell_at(os + tb * ds, los, inv_hs, dim_s);
            if (sb != sa) {
                const float tc = fminf(fmaxf((los + (float)(sb > sa ? sa + 1 : sa) * hs - os) * __fdividef(1.f, ds), ta), tb);
                if (second) {
                    cs = sb > sa ? sa + 1 : sa - 1;
                    t_enter = ta = tc;
                } else {
                    t_end = tb = tc;
                }
            } else if (second) {
                return 0u;
            }
        }
        cx = along_y ? cs : c;
        cy = along_y ? c : cs;
    }
    const float lo_z = fine ? S.f_lo.z : S.g_lo.z, inv_hz = fine ? S.f_inv_h.z : S.g_inv_h.z;
    const int dim_y = fine ? S.f_dim.y : S.g_dim.y, dim_z = fine ? S.f_dim.z : S.g_dim.z;
    const uint32_t *cs = fine ? S.f_cell_start : S.cell_start;
    const float za = fmaf(t_enter, d.z, o.z), zb = fmaf(tb, d.z, o.z);
    const int cza = cell_at(fminf(za, zb) - S.g_rm, lo_z, inv_hz, dim_z);
    const int czb = cell_at(fmaxf(za, zb) + S.g_rm, lo_z, inv_hz, dim_z);
    const uint32_t col = ((uint32_t)cx * (uint32_t)dim_y + (uint32_t)cy) * (uint32_t)dim_z;
    begin = cs[col + (uint32_t)cza];
    return cs[col + (uint32_t)czb + 1u] - begin;
}

template <bool DBG>
__device__ __forceinline__ void end_ray(const TraceP &P, Lane &R, int reason, Counters &cn) {
    if (DBG && P.path_hash) P.path_hash[P.items[R.item].hash_begin + R.i] = fnv_step(R.h, 0x20000u | (uint32_t)reason);
    cn.rays++;
    R.state = kNeedRay;
}

// Emission (Eq. 6) of ray i of item `item` (a transmit of one scene) from element e.
// With transmit mixing the ray first draws its transmit (Sec. 2.3); a synthetic-
// aperture transmit emits every ray from its one element.
template <bool DBG, bool EXT, int GEO>
__device__ __forceinline__ void start_ray(const TraceP &P, Lane &R, uint32_t item, const ItemP &slot_item,
                                          uint32_t i, uint32_t e, Counters &cn) {
    constexpr bool CVX = (GEO & kGeoConvex) != 0, EMIT = EXT && (GEO & kGeoEmit) != 0;
    if (EMIT && P.mix_tx > 0) {
        const uint4 y = philox(make_uint4(i, 0u, 0u, 1u), P.key);
        item = (uint32_t)(((uint64_t)(y.x >> 8) * (uint64_t)P.mix_tx) >> 24);
    }
    const ItemP &IT = EMIT && P.mix_tx > 0 ? P.items[item] : slot_item;
    if (EMIT && IT.kind == UR_TX_SYNTHETIC) e = (uint32_t)IT.vx;
    const uint4 x = draw<EXT>(make_uint4(i, IT.stream, 0u, 0u), P.key);
    const float xe = fmaf((float)e, P.pitch, P.x_first);
    R.o = make_float3(fmaf(u24(x.x) - 0.5f, P.pitch, xe), (u24(x.y) - 0.5f) * P.H, 0.f);
    float arc_s = 0.f, arc_h = 0.f;             // convex: sines of the point's arc angle and of half of it
    float3 nrm = make_float3(0.f, 0.f, 1.f);   // normal at the emission point
    if (CVX) {                                  // a point of the element's arc face
        const float ph = fmaf((float)e + u24(x.x) - 0.5f, P.dphi, P.phi0);
        float sn, cs, sh, ch;
        sincosf(ph, &sn, &cs);
        sincosf(0.5f * ph, &sh, &ch);
        nrm = make_float3(sn, 0.f, cs);
        arc_s = sn;
        arc_h = sh;
        R.o = make_float3(__fmul_rn(P.radius, sn), R.o.y, __fmul_rn(-2.f * P.radius * sh, sh));
    }
    if (!EXT || IT.kind == UR_TX_PLANE) {
        R.d = make_float3(IT.sin_t, 0.f, IT.cos_t);
    } else if (EMIT && IT.kind == UR_TX_SYNTHETIC) {   // uniform angle to the face normal in (-pi/2, pi/2)
        const float th = ((float)(int)((x.z >> 8) - (1u << 23)) + 0.5f) * (kPiF * 0x1p-24f);
        float st, ct;
        sincosf(th, &st, &ct);
        R.d = make_float3(sum2(nrm.x, ct, nrm.z, st), 0.f, sum2(nrm.z, ct, -nrm.x, st));
    } else {   // along the line from the virtual source, or toward the focus, in the xz plane
        const float sg = IT.kind == UR_TX_DIVERGING ? 1.f : -1.f;
        const float dx = sg * (CVX ? fmaf(P.radius, arc_s, -IT.vx) : R.o.x - IT.vx);
        const float dz = sg * (CVX ? fmaf(-2.f * P.radius * arc_h, arc_h, -IT.vz) : R.o.z - IT.vz);
        const float l = sqrtf(sum2(dx, dx, dz, dz));
        R.d = make_float3(dx / l, 0.f, dz / l);
    }
    R.t = P.delay[(uint32_t)IT.angle * (uint32_t)P.n_el + e];
    R.w = (EXT ? dot3(R.d, nrm) : R.d.z) * IT.inv_n;   // Eq. 6: cosine to the face normal over N
    R.scene = IT.scene;
    R.med = scene_of<GEO>(P, IT.scene).med_array;
    R.b = 0;
    R.prev = -1;
    R.L = 0.f;
    R.i = i;
    R.item = item;
    R.stream = IT.stream;
    R.h = kFnvOffset;
    R.mis = false;
    if (EXT && !(R.w > 0.f)) {   // aimed into a convex probe: no ray
        end_ray<DBG>(P, R, kEndArrayMiss, cn);
        return;
    }
    R.state = kNeedSeg;
}

// Secondary ray of a rough vertex to a uniformly drawn element centre, weighted
// against BSDF sampling of the same direction by the balance heuristic.
template <bool DBG, bool REC, int GEO>
__device__ void rough_connection(const TraceP &P, const SceneP &S, const Lane &R, float3 n, int m2, float a2,
                                 Counters &cn) {
    constexpr bool CVX = (GEO & kGeoConvex) != 0, MESH = (GEO & kGeoMesh) != 0;
    const uint4 x = philox(make_uint4(R.i, R.stream, 4u | ((uint32_t)R.b << 8), 0u), P.key);
    const uint32_t e = (uint32_t)(((uint64_t)(x.x >> 8) * (uint64_t)P.n_el) >> 24);
    float3 ce, ne;
    elem_frame<CVX>(P, e, ce, ne);
    const float3 v = ce - R.o;
    const float D = sqrtf(dot3_yx(v, v));
    const float3 o = make_float3(v.x / D, v.y / D, v.z / D);
    const float cos_e = CVX ? -dot3(o, ne) : -o.z;   // at the element, to its normal (+z on a linear array)
    const float fd = CVX ? directivity(P, -dot3(v, ne), cross2(v, ne)) : directivity(P, -v.z, sum2(v.y, v.y, v.x, v.x));
    if (!(fd > 0.f)) return;
    const Medium &M = S.med[R.med], &M2 = S.med[m2];
    float pdf;
    const float f = rough_eval(R.d, n, o, a2, M, M2, pdf);
    if (!(f > 0.f)) return;
    cn.connections++;
    ff tc;
    float att;
    const float fac = connection_to<MESH>(S, R.o, dot3(o, n) > 0.f ? R.med : m2, R.hit, ce, tc, att);
    if (fac == 0.f) return;
    const ff ta = ff_add(R.t, tc);
    if (ff_gt(ta, P.t_last)) return;
    const float omega = P.pitch * P.H * cos_e / (D * D);   // element solid angle seen from the vertex
    const float p_nee = 1.f / ((float)P.n_el * omega);
    const float amp = R.w * f * fd * fac * expf(-att) / (p_nee + pdf);
    emit<DBG, REC>(P, R.item * (uint32_t)P.n_el + e, ta, amp, R.i,
                   0x80000000u | ((uint32_t)R.b << 24) | (uint32_t)(R.hit + 1));
    cn.arrivals++;
}

// Microfacet sampling at a rough vertex: normal from D(m)(m.n), the smooth branch
// about it, weight |i.m| G / (|i.n| |m.n|).  Returns false if the sample is not
// admissible (back-facing microfacet or a direction on the wrong side).
__device__ bool rough_scatter(const TraceP &P, const SceneP &S, Lane &R, float3 n, int m2, float a2,
                              uint32_t &branch) {
    const float cos_i = -dot3(n, R.d);
    const uint4 x = philox(make_uint4(R.i, R.stream, 3u | ((uint32_t)R.b << 8), 0u), P.key);
    float mn;   // m.n, the sampled cosine (exact where a dot product would cancel for grazing m)
    const float3 m = ggx_sample(n, a2, u24(x.x), u24(x.y), mn);
    const float c_im = -dot3(R.d, m);
    if (!(c_im > 0.f)) return false;
    const Medium &M = S.med[R.med], &M2 = S.med[m2];
    float r, cos_t;
    const bool tir = !fresnel(c_im, M.c, M.Z, M2.c, M2.Z, r, cos_t);
    float3 o;
    float fac, pb, jac;
    bool far = false;
    if (tir) {
        branch = 2;
        o = unit3(along(R.d, 2.f * c_im, m));
        fac = 1.f;
        pb = 1.f;
        jac = 0.25f / c_im;
    } else {
        const uint4 y = philox(make_uint4(R.i, R.stream, 1u | ((uint32_t)R.b << 8), 0u), P.key);
        const float Rs = r * r;
        if (u24(y.x) < Rs) {
            branch = 0;
            o = unit3(along(R.d, 2.f * c_im, m));
            fac = r / Rs;
            pb = Rs;
            jac = 0.25f / c_im;
        } else {
            branch = 1;
            const float eta = M2.c / M.c;
            o = unit3(blend(eta, R.d, fmaf(eta, c_im, -cos_t), m));
            pb = transmitted(c_im, cos_t, M.Z, M2.Z);
            fac = 1.f / sqrtf(pb);
            const float om = dot3(o, m);
            const float den = fmaf(eta, c_im, om);
            jac = -om / (den * den);
            far = true;
        }
    }
    const float on = dot3(o, n);
    if (far ? !(on < 0.f) : !(on > 0.f)) return false;
    const float G = ggx_g1(cos_i, a2) * ggx_g1(fabsf(on), a2);
    R.w *= fac * c_im * G / (cos_i * mn);
    R.mis = true;
    R.mp = R.o;
    R.mpdf = ggx_d(mn, a2) * mn * jac * pb;
    R.d = o;
    if (far) R.med = m2;
    return true;
}

// End of a segment: time of flight and attenuation along it, then the array
// plane (aperture return), the absorbing bottom, the time window, the bounce
// budget, or a boundary interaction (Eqs. 7-11) and the next segment.
template <bool DBG, bool SPLIT, bool REC, bool ROUGH, int GEO>
__device__ void finish_segment(const TraceP &P, Lane &R, Counters &cn) {
    constexpr bool CVX = (GEO & kGeoConvex) != 0, MESH = (GEO & kGeoMesh) != 0;
    const SceneP &S = scene_of<GEO>(P, R.scene);
    const Medium &M = S.med[R.med];
    R.t = ff_add(R.t, ff_mul_f(R.seg, M.slow));
    R.w *= expf(-M.a * R.seg);
    R.L += R.seg;
    R.o = along(R.o, R.seg, R.d);
    if (R.clipped) {
        end_ray<DBG>(P, R, kEndPath, cn);
        return;
    }
    if (CVX && R.hit == S.n_bnd + 2) {   // passed beside a convex probe
        end_ray<DBG>(P, R, kEndArrayMiss, cn);
        return;
    }
    if (R.hit == S.n_bnd) {  // array surface: only paths returning to the aperture are kept
        int el = -1;
        if (CVX) {   // the probe's cylinder: the element whose arc holds the hit
            const float u = (atan2f(R.o.x, R.o.z + P.radius) - P.phi0) / P.dphi + 0.5f;
            if (fabsf(R.o.y) <= 0.5f * P.H && u >= 0.f && u < (float)P.n_el) el = min((int)floorf(u), P.n_el - 1);
        } else {
            R.o.z = 0.f;
            const float xl = fmaf(-0.5f, P.pitch, P.x_first);
            if (fabsf(R.o.y) <= 0.5f * P.H && R.o.x >= xl && R.o.x < fmaf((float)P.n_el, P.pitch, xl)) {
                el = (int)floorf((R.o.x - xl) / P.pitch);
                if (el > P.n_el - 1) el = P.n_el - 1;
            }
        }
        int reason = kEndArrayMiss;
        if (el >= 0) {
            float3 ce = make_float3(0.f, 0.f, 0.f), ne = make_float3(0.f, 0.f, 1.f);
            if (ROUGH) elem_frame<CVX>(P, (uint32_t)el, ce, ne);
            const float fd = CVX ? directivity(P, -dot3(R.d, ne), cross2(R.d, ne))
                           : directivity(P, -R.d.z, ROUGH ? sum2(R.d.y, R.d.y, R.d.x, R.d.x) : sum2(R.d.x, R.d.x, R.d.y, R.d.y));
            if (fd > 0.f && !ff_gt(R.t, P.t_last)) {
                float wa = R.w * fd;
                if (ROUGH && R.mis) {   // balance heuristic against the rough vertex's secondary ray
                    const float3 v = ce - R.mp;
                    const float D2 = dot3_yx(v, v);
                    const float omega = P.pitch * P.H * ((CVX ? -dot3(v, ne) : -v.z) / sqrtf(D2)) / D2;
                    if (omega > 0.f) wa *= 1.f / (1.f + 1.f / ((float)P.n_el * omega * R.mpdf));
                }
                emit<DBG, REC>(P, R.item * (uint32_t)P.n_el + (uint32_t)el, R.t, wa, R.i,
                          0x80000000u | ((uint32_t)R.b << 24));
                cn.arrivals++;
            }
            reason = kEndAperture;
        }
        end_ray<DBG>(P, R, reason, cn);
        return;
    }
    if (R.hit == S.n_bnd + 1) {
        end_ray<DBG>(P, R, kEndBottom, cn);
        return;
    }
    const bool on_tri = MESH && R.hit >= S.tri_base;
    if (!on_tri && S.bnd[R.hit].kind == kPlaneZ) R.o.z = S.bnd[R.hit].p[0];
    if (ff_gt(R.t, P.t_last)) {
        end_ray<DBG>(P, R, kEndTime, cn);
        return;
    }
    if (R.b >= P.max_b) {
        end_ray<DBG>(P, R, kEndMaxB, cn);
        return;
    }
    float3 n_out;
    int m_neg, m_pos;
    float alpha;
    if (on_tri) {
        surface_tri(S, R.hit, n_out, m_neg, m_pos, alpha);
    } else {
        const Bnd &B = S.bnd[R.hit];
        n_out = outward(B, R.o);
        m_neg = B.med_neg;
        m_pos = B.med_pos;
        alpha = B.alpha;
    }
    const float dn = dot3(R.d, n_out);
    const int m2 = dn > 0.f ? m_pos : m_neg;
    const float3 n = dn > 0.f ? make_float3(-n_out.x, -n_out.y, -n_out.z) : n_out;
    if (ROUGH && alpha > 0.f) {   // rough boundary: secondary ray first, then the BSDF sample
        const float a2 = alpha * alpha;
        rough_connection<DBG, REC, GEO>(P, S, R, n, m2, a2, cn);
        cn.interactions++;
        uint32_t rb = 0;
        if (!rough_scatter(P, S, R, n, m2, a2, rb)) {
            end_ray<DBG>(P, R, kEndRough, cn);
            return;
        }
        if (DBG) R.h = fnv_step(R.h, 0x10000u | ((uint32_t)R.hit << 4) | rb);
        R.b += 1;
        R.prev = R.hit;
        R.state = kNeedSeg;
        return;
    }
    const float cos_i = -dot3(n, R.d);
    const float3 dr = unit3(along(R.d, 2.f * cos_i, n));
    const Medium &M2 = S.med[m2];
    float r, cos_t, Rs, rs, cts = 0.f;
    bool tir;
    uint32_t branch;
    if (!SPLIT) {   // the media decide their own branches
        tir = !fresnel(cos_i, M.c, M.Z, M2.c, M2.Z, r, cos_t);
        Rs = r * r;
    } else {        // frozen sampling media decide the branch and its probability
        tir = !fresnel(cos_i, S.cs[R.med], S.Zs[R.med], S.cs[m2], S.Zs[m2], rs, cts) ||
              !fresnel(cos_i, M.c, M.Z, M2.c, M2.Z, r, cos_t);
        Rs = rs * rs;
    }
    if (tir) {
        branch = 2;
        R.d = dr;
    } else {
        const uint4 y = draw<ROUGH>(make_uint4(R.i, R.stream, 1u | ((uint32_t)R.b << 8), 0u), P.key);
        if (u24(y.x) < Rs) {
            branch = 0;
            R.w *= r / Rs;
            R.d = dr;
        } else {
            branch = 1;
            const float eta = M2.c / M.c;
            // 1 - R as 4 Z1 Z2 cos_i cos_t / (Z2 cos_i + Z1 cos_t)^2: no cancellation near the critical angle
            const float T = transmitted(cos_i, cos_t, M.Z, M2.Z);
            R.w *= SPLIT ? sqrtf(T) / transmitted(cos_i, cts, S.Zs[R.med], S.Zs[m2]) : rsqrtf(T);
            R.d = unit3(blend(eta, R.d, fmaf(eta, cos_i, -cos_t), n));
            R.med = m2;
        }
    }
    cn.interactions++;
    if (ROUGH && branch != 1) R.mis = false;   // a smooth reflection: the secondary ray cannot produce this path
    if (DBG) R.h = fnv_step(R.h, 0x10000u | ((uint32_t)R.hit << 4) | branch);
    R.b += 1;
    R.prev = R.hit;
    R.state = kNeedSeg;
}

// A queued scatterer event: element drawn uniformly (Philox keyed by ray,
// transmit, segment and scatterer) and the receive directivity (Eq. 13).  An
// event the element receives goes on to the warp's connection ring with its
// arrival time and amplitude so far (the connection ray's part follows there).
template <bool EXT, int GEO>
__device__ __forceinline__ bool event_element(const TraceP &P, const WarpQueue &Q, int slot, uint32_t &e, ff &t_pre,
                                              float &amp_pre) {
    constexpr bool CVX = (GEO & kGeoConvex) != 0;
    const uint32_t ray = Q.ray[slot], kmb = Q.kmb[slot], j = Q.j[slot];
    const float tca = Q.tca[slot], w = Q.w[slot];
    const ff t = {Q.t_hi[slot], Q.t_lo[slot]};
    const uint32_t item = kmb >> 16;
    const int med = (int)((kmb >> 8) & 0xffu), b = (int)(kmb & 0xffu);
    const ItemP &IT = P.items[item];
    const SceneP &S = scene_of<GEO>(P, IT.scene);
    const float4 q = S.scat[j];
    const uint4 x = draw<EXT>(make_uint4(ray, IT.stream, 2u | ((uint32_t)b << 8), j), P.key);
    e = (uint32_t)(((uint64_t)(x.x >> 8) * (uint64_t)P.n_el) >> 24);
    float fd;
    if (CVX) {   // convex array: directivity to the element's normal
        float3 ce, ne;
        elem_frame<CVX>(P, e, ce, ne);
        const float3 v = make_float3(q.x - ce.x, q.y - ce.y, q.z - ce.z);
        fd = directivity(P, dot3(v, ne), cross2(v, ne));
    } else {
        const float vx = fmaf((float)e, P.pitch, P.x_first) - q.x;
        fd = directivity(P, q.z, sum2(vx, vx, q.y, q.y));
    }
    if (!(fd > 0.f)) return false;
    const Medium &M = S.med[med];
    t_pre = ff_add(t, ff_mul_f(tca, M.slow));
    amp_pre = w * expf(-M.a * tca) * q.w * (float)P.n_el * fd;
    return true;
}

// Scatterer events waiting for their connection ray to the drawn element, one ring per warp (SoA).
struct ConnQueue {
    uint32_t ray[kQueue], kmb[kQueue], j[kQueue], e[kQueue];
    float t_hi[kQueue], t_lo[kQueue], amp[kQueue];
};

// A queued connection: the straight ray from the scatterer to the element centre,
// its transmission factors, time and attenuation; the arrival goes to the queue.
template <bool DBG, bool REC, bool EXT, int GEO>
__device__ __forceinline__ void process_connection(const TraceP &P, const ConnQueue &C, int slot, Counters &cn) {
    constexpr bool CVX = (GEO & kGeoConvex) != 0, MESH = (GEO & kGeoMesh) != 0;
    const uint32_t ray = C.ray[slot], kmb = C.kmb[slot], j = C.j[slot], e = C.e[slot];
    const uint32_t item = kmb >> 16;
    const int med = (int)((kmb >> 8) & 0xffu), b = (int)(kmb & 0xffu);
    const ItemP &IT = P.items[item];
    const SceneP &S = scene_of<GEO>(P, IT.scene);
    const float4 q = S.scat[j];
    cn.connections++;
    ff tc;
    float att, fac;
    if (CVX) {
        float3 ce, ne;
        elem_frame<CVX>(P, e, ce, ne);
        fac = connection_to<MESH>(S, make_float3(q.x, q.y, q.z), med, -1, ce, tc, att);
    } else {
        fac = connection<MESH>(S, make_float3(q.x, q.y, q.z), med, -1, fmaf((float)e, P.pitch, P.x_first), tc, att);
    }
    if (fac == 0.f) return;
    const ff ta = ff_add({C.t_hi[slot], C.t_lo[slot]}, tc);
    if (ff_gt(ta, P.t_last)) return;
    const float amp = C.amp[slot] * fac * expf(-att);
    emit<DBG, REC>(P, item * (uint32_t)P.n_el + e, ta, amp, ray, ((uint32_t)b << 24) | j);
    cn.arrivals++;
}

// Events [qhead + lane] for the lanes below n: element draw and directivity; the ones the
// element receives join the connection ring, which is traced 32 at a time with all lanes.
template <bool DBG, bool REC, bool EXT, int GEO>
__device__ __forceinline__ void drain_events(const TraceP &P, const WarpQueue &Q, ConnQueue &CQ, int qhead, int n,
                                             int &chead, int &cn_q, Counters &cn) {
    const int lane = threadIdx.x & 31;
    uint32_t e = 0;
    ff t_pre = {0.f, 0.f};
    float amp_pre = 0.f;
    const int slot = (qhead + lane) & (kQueue - 1);
    const bool go = lane < n && event_element<EXT, GEO>(P, Q, slot, e, t_pre, amp_pre);
    const unsigned m = __ballot_sync(0xffffffffu, go);
    if (go) {
        const int c = (chead + cn_q + __popc(m & ((1u << lane) - 1u))) & (kQueue - 1);
        CQ.ray[c] = Q.ray[slot];
        CQ.kmb[c] = Q.kmb[slot];
        CQ.j[c] = Q.j[slot];
        CQ.e[c] = e;
        CQ.t_hi[c] = t_pre.hi;
        CQ.t_lo[c] = t_pre.lo;
        CQ.amp[c] = amp_pre;
    }
    cn_q += __popc(m);
    if (cn_q >= 32) {
        __syncwarp();
        process_connection<DBG, REC, EXT, GEO>(P, CQ, (chead + lane) & (kQueue - 1), cn);
        __syncwarp();
        chead = (chead + 32) & (kQueue - 1);
        cn_q -= 32;
    }
}

// Inclusive prefix sum over the warp's lanes.
__device__ __forceinline__ uint32_t prefix_sum(uint32_t x) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
        if ((int)(threadIdx.x & 31) >= off) x += y;
    }
    return x;
}

// Runs of numbered items: this lane's run of `count` begins `off` items into the current batch of 32
// (unsigned: earlier runs wrap to large values).  Returns, for the lane-th item of the batch, the
// rank of its run among the runs that are not empty; `seen` counts those begun in earlier batches.
__device__ __forceinline__ uint32_t owner_rank(uint32_t off, uint32_t count, uint32_t &seen) {
    const unsigned begins = __reduce_or_sync(0xffffffffu, count && off < 32u ? 1u << off : 0u);
    const uint32_t rank = seen + (uint32_t)__popc(begins & (lanemask_lt() * 2u + 1u)) - 1u;
    seen += (uint32_t)__popc(begins);
    return rank;
}

__device__ __forceinline__ float3 shfl3(float3 v, int lane) {
    return make_float3(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane),
                       __shfl_sync(0xffffffffu, v.z, lane));
}

// The item whose slot range holds `slot` (item slot ranges are pool-aligned and ascending).
__device__ __forceinline__ uint32_t item_of(const TraceP &P, uint64_t slot) {
    int lo = 0, hi = P.n_items - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.items[mid].slot_begin <= slot) lo = mid; else hi = mid - 1;
    }
    return (uint32_t)lo;
}

// Residency, trading warps for registers, measured (us) at 2, 3 and 4 CTAs per SM: plane waves in one
// scene (constants free the registers of its fields) 3 (layered frame 3522 against 3789 at 4, one
// 7-degree wave the same), batches of several scenes 4 (21.9 ms against 23.0 at 3), extended 3 (paper
// settings 4773, 4200, 4910; diverging 2170, 1790, 2090), meshes 3 (mesh bone 7055, 6573, 7446).  The
// grid is sized for 4 CTAs per SM: CTAs that find the ray pools empty exit at once.
template <bool ROUGH, int GEO>
constexpr int trace_ctas_per_sm() { return ROUGH || (GEO & kGeoOne) ? 3 : 4; }

// Lanes without a ray before a warp starts new ones.  Measured (us) at 10, 14, 18: layered frame 3532,
// 3495, 3452, two scenes x 16 plane waves 18963, 18766, 18685; paper settings 4208, 4380, 4428, mesh bone
// 6597, 6625, 6640 (1 and 4: layered frame 4031 and 3908 against 3761 at 10, paper settings alike).
constexpr int kIdleMin = 18, kIdleMinExtended = 10;

// Persistent tracer.  Each iteration of the warp's loop (1) takes one step of every lane's path
// (finish the segment, start a new ray in idle lanes, set up the next segment), (2) makes the
// column visits of all 32 segments, numbered across the warp and made 32 at a time, and tests the
// references of 32 visits the same way, (3) hands scatterer events to a per-warp queue that is
// drained 32 events at a time; the events the drawn element receives wait in a second ring for
// their connection rays, traced 32 at a time as well.  Every stage runs with (nearly) all lanes: a
// segment's walk has no state of its own, its k-th visit is computed from the segment.  Ray slots
// are element-major: a freshly claimed batch of lanes traces neighbouring rays of one element;
// slot -> ray i = m * n_el + e.
//
// Bound by instruction issue (61 % of cycles) and the latency of reference loads.  Before, each lane
// walked its own segment, one column per iteration, and segments were finished once 20 lanes
// waited: 425 warp instructions per ray of the layered frame with 21.7 of 32 lanes; this way about
// 300 with 26.3.  Trace, in us before, with this and with the cells, residency and threshold that suit it: layered
// frame (1e7 rays, 0 degrees) 5578, 4020, 3453; paper settings 5960, 4860, 4225; 9 diverging waves 3050,
// 1940, 1798; mesh bone (25 x 256k rays) 10660, 7560, 6557; two scenes x 16 plane waves x 1e6 rays 29.3,
// 19.7, 18.7 ms.  The warp synchronisations after the divergent steps keep the lanes together (mesh
// bone 8610 -> 7760 us, paper settings 4920 -> 4630).
template <bool DBG, bool SPLIT, bool REC, bool ROUGH, int GEO>
__global__ void __launch_bounds__(kBlock, trace_ctas_per_sm<ROUGH, GEO>()) k_trace(const __grid_constant__ TraceP P) {
    __shared__ WarpQueue s_q[kWarps];
    __shared__ ConnQueue s_c[kWarps];
    __shared__ WarpVisits s_v[kWarps];
    WarpQueue &Q = s_q[threadIdx.x >> 5];
    WarpVisits &V = s_v[threadIdx.x >> 5];
    ConnQueue &CQ = s_c[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const uint64_t n_slots = P.n_slots;
    const int idle_min = P.resolve_batch > 0 ? P.resolve_batch : ROUGH ? kIdleMinExtended : kIdleMin;
    Counters cn = {0, 0, 0, 0, 0, 0};
    Lane R;
    R.state = kNeedRay;
    uint64_t pool_next = 0;
    uint32_t pool_cnt = 0, pool_item = 0;
    bool pool_dry = false;
    int qhead = 0, qn = 0;     // warp-uniform ring bookkeeping: scatterer events
    int chead = 0, cqn = 0;    // and connections

    for (;;) {
        // (1) one step of every lane's path
        if (R.state == kHasSeg) finish_segment<DBG, SPLIT, REC, ROUGH, GEO>(P, R, cn);
        __syncwarp();
        unsigned need = __ballot_sync(0xffffffffu, R.state == kNeedRay);
        if (need && (__popc(need) >= idle_min || __ballot_sync(0xffffffffu, R.state == kNeedSeg) == 0u)) {
            uint64_t my_slot = ~0ull;
            while (need) {
                if (pool_cnt == 0) {
                    if (!pool_dry) {
                        unsigned long long base = 0;
                        if (lane == 0) base = atomicAdd(P.next_slot, (unsigned long long)kPool);
                        base = __shfl_sync(0xffffffffu, base, 0);
                        pool_next = base;
                        pool_cnt = base >= n_slots ? 0u : (uint32_t)kPool;
                        pool_dry = pool_cnt == 0;
                        if (!pool_dry) pool_item = item_of(P, base);
                    }
                    if (pool_dry) {
                        if (R.state == kNeedRay && my_slot == ~0ull) R.state = kFinished;
                        break;
                    }
                }
                const uint32_t take = min((uint32_t)__popc(need), pool_cnt);
                const uint32_t rank = (uint32_t)__popc(need & lanemask_lt());
                if (((need >> lane) & 1u) && rank < take) my_slot = pool_next + rank;
                pool_next += take;
                pool_cnt -= take;
                need = __ballot_sync(0xffffffffu, R.state == kNeedRay && my_slot == ~0ull);
            }
            if (my_slot != ~0ull) {
                // A warp that used up a pool and claimed the next one in the same pass holds slots
                // of both; a slot before the current item's range belongs to an earlier item.
                uint32_t item = pool_item;
                if (my_slot < P.items[item].slot_begin) item = item_of(P, my_slot);
                const ItemP &IT = P.items[item];
                const uint64_t local = my_slot - IT.slot_begin;
                if (ROUGH && (GEO & kGeoEmit) && P.mix_list) {   // a mixed sequence in (drawn transmit, element) order
                    if (local < IT.n_rays) {
                        const uint32_t i = P.mix_list[local];
                        start_ray<DBG, ROUGH, GEO>(P, R, item, IT, i, i % (uint32_t)P.n_el, cn);
                    }
                } else {
                    const uint32_t m = (uint32_t)(local % IT.rays_per_el);
                    const uint64_t e = local / IT.rays_per_el;
                    const uint32_t i = m * (uint32_t)P.n_el + (uint32_t)e;
                    if (e < (uint64_t)P.n_el && i < IT.n_rays) start_ray<DBG, ROUGH, GEO>(P, R, item, IT, i, (uint32_t)e, cn);
                }
            }
        }
        __syncwarp();
        uint32_t n_vis = 0u;
        if (R.state == kNeedSeg) n_vis = start_segment<GEO, !ROUGH>(P, R, cn);
        __syncwarp();
        if (__all_sync(0xffffffffu, R.state == kFinished)) break;

        // (2) the column visits of all lanes' segments, numbered across the warp (prefix sum of
        // their counts) and made 32 at a time; the references of 32 visits are numbered and tested
        // the same way, each lane reading its reference's ray from the owning lane's registers
        const uint32_t v_incl = prefix_sum(n_vis), v_first = v_incl - n_vis;
        const uint32_t v_total = __shfl_sync(0xffffffffu, v_incl, 31);
        const uint32_t kmb = (R.item << 16) | ((uint32_t)R.med << 8) | (uint32_t)R.b;
        const unsigned v_owners = __ballot_sync(0xffffffffu, n_vis > 0u);
        if (n_vis) V.seg_lane[__popc(v_owners & lanemask_lt())] = (uint32_t)lane;
        __syncwarp();
        uint32_t v_seen = 0;   // segments whose visits began in earlier batches
        for (uint32_t v_base = 0; v_base < v_total; v_base += 32) {
            const uint32_t kv = v_base + (uint32_t)lane;
            const int so = (int)V.seg_lane[owner_rank(v_first - v_base, n_vis, v_seen)];   // the lane whose segment visit kv belongs to
            const uint32_t first = __shfl_sync(0xffffffffu, v_first, so), n = __shfl_sync(0xffffffffu, n_vis, so);
            const float3 vo = shfl3(R.o, so), vd = shfl3(R.d, so);
            const float t0 = __shfl_sync(0xffffffffu, R.t0, so), t1 = __shfl_sync(0xffffffffu, R.t1, so);
            const float seg = __shfl_sync(0xffffffffu, R.seg, so);
            const uint32_t walk = __shfl_sync(0xffffffffu, R.walk, so);
            const int v_scene = (GEO & kGeoOne) ? 0 : __shfl_sync(0xffffffffu, R.scene, so);
            uint32_t cnt = 0, begin = 0;
            float v_lo = 0.f, v_hi = 0.f;
            if (kv < v_total)
                cnt = column_visit<!ROUGH>(scene_of<GEO>(P, v_scene), vo, vd, walk, t0, t1, seg, kv - first, n, begin, v_lo, v_hi);
            const uint32_t incl = prefix_sum(cnt), excl = incl - cnt;
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            const unsigned owners = __ballot_sync(0xffffffffu, cnt > 0u);
            __syncwarp();
            if (cnt)
                V.visit[__popc(owners & lanemask_lt())] =
                    make_uint4((uint32_t)so | (walk & kWalkFine), begin - excl, __float_as_uint(v_lo), __float_as_uint(v_hi));
            __syncwarp();
            uint32_t seen = 0;   // visits whose references began in earlier batches
            for (uint32_t base = 0; base < total; base += 32) {
                const uint32_t k = base + (uint32_t)lane;
                const uint4 vis = V.visit[owner_rank(excl - base, cnt, seen)];   // the visit that holds reference k
                const int ray_lane = (int)(vis.x & 31u);
                bool cand = false;
                float tca = 0.f;
                uint32_t j = 0;
                const float3 A = shfl3(R.o, ray_lane), B = shfl3(R.d, ray_lane);
                const int scene = (GEO & kGeoOne) ? 0 : __shfl_sync(0xffffffffu, R.scene, ray_lane);
                if (k < total) {
                    const SceneP &S = scene_of<GEO>(P, scene);
                    const float4 *refs = !ROUGH && (vis.x & kWalkFine) ? S.f_refs : S.refs;
                    const float4 q = refs[vis.y + k];
                    const float3 v = make_float3(q.x - A.x, q.y - A.y, q.z - A.z);
                    tca = dot3(v, B);
                    if (tca > 0.f && tca >= __uint_as_float(vis.z) && tca < __uint_as_float(vis.w)) {
                        const float3 pe = along(v, -tca, B);
                        cand = dot3(pe, pe) < S.r2;
                        j = __float_as_uint(q.w);
                        if (cand) cn.candidates++;
                        // An event no element can receive (Eq. 13: farther across than the cutoff for
                        // every element of a linear array, by its y alone) needs no element drawn.  The
                        // same products as directivity(), whose y^2 + x^2 is rounded up from y^2.
                        if (!(GEO & kGeoConvex) && q.y * q.y > P.t2ac * (q.z * q.z)) cand = false;
                    }
                }
                const unsigned m = __ballot_sync(0xffffffffu, cand);
                if (m) {
                    const uint32_t e_ray = __shfl_sync(0xffffffffu, R.i, ray_lane), e_kmb = __shfl_sync(0xffffffffu, kmb, ray_lane);
                    const float e_thi = __shfl_sync(0xffffffffu, R.t.hi, ray_lane), e_tlo = __shfl_sync(0xffffffffu, R.t.lo, ray_lane);
                    const float e_w = __shfl_sync(0xffffffffu, R.w, ray_lane);
                    if (cand) {
                        const int slot = (qhead + qn + __popc(m & lanemask_lt())) & (kQueue - 1);
                        Q.ray[slot] = e_ray;
                        Q.kmb[slot] = e_kmb;
                        Q.j[slot] = j;
                        Q.tca[slot] = tca;
                        Q.t_hi[slot] = e_thi;
                        Q.t_lo[slot] = e_tlo;
                        Q.w[slot] = e_w;
                    }
                    qn += __popc(m);
                    if (qn >= 32) {
                        __syncwarp();
                        drain_events<DBG, REC, ROUGH, GEO>(P, Q, CQ, qhead, 32, chead, cqn, cn);
                        __syncwarp();
                        qhead = (qhead + 32) & (kQueue - 1);
                        qn -= 32;
                    }
                }
            }
        }
    }
    // (3) drain the queues
    __syncwarp();
    drain_events<DBG, REC, ROUGH, GEO>(P, Q, CQ, qhead, qn, chead, cqn, cn);
    __syncwarp();
    if (lane < cqn) process_connection<DBG, REC, ROUGH, GEO>(P, CQ, (chead + lane) & (kQueue - 1), cn);

    if (P.stats) {
        const uint32_t v[6] = {cn.rays, cn.segments, cn.interactions, cn.candidates, cn.connections, cn.arrivals};
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const uint32_t s = __reduce_add_sync(0xffffffffu, v[c]);
            if (lane == 0 && s) atomicAdd(&P.stats[c], (unsigned long long)s);
        }
    }
}

}  // namespace

// Variants with frozen sampling media, with recorded (ray, event) words and the
// extended variants (rough boundaries, diverging and focused transmits; one per
// geometry: linear or convex array, with or without triangle meshes; with or
// without synthetic-aperture emission and transmit mixing, whose code cost the
// rough layered frame 6 % and the paper-settings acquisition 9 % when every
// extended trace carried it) are compiled separately so the usual kernel carries
// none of their code.  Mesh variants always carry the emission
// code.  The extended variants never record or freeze sampling media (the adjoint and
// ur_scene_set_media refuse such scenes and transmits).
template <int GEO>
void launch_extended(const TraceP &P, bool debug, int block, int grid, cudaStream_t s);

}  // namespace ur
