// Device building blocks of the fitness path shared by its kernels (the
// cluster-bitmap kernel in raster.cu and the binned pipeline in binned.cu):
// per-candidate kinematics in double-float arithmetic (Sec. III-A.2,
// III-A.3), compensated FP32 projection with the 1/256 px snap, integer
// triangle set-up and the top-left-rule raster primitives, and the keypoint
// term of Eq. kpts_loss.
#pragma once

#include "cma_device.cuh"
#include "df.cuh"

namespace trk {

// ----------------------------------------------------------------------------
// Per-candidate kinematics in double-float arithmetic (Sec. III-A.2, III-A.3)
// ----------------------------------------------------------------------------
__device__ __forceinline__ dfl dfc(float2 v) { return {v.x, v.y}; }

__device__ __forceinline__ dfl dot3(dfl a0, dfl b0, dfl a1, dfl b1, dfl a2, dfl b2)
{
    return df_add(df_add(df_mul(a0, b0), df_mul(a1, b1)), df_mul(a2, b2));
}

// Entry (i, j) of the elementary rotation about axis x/y/z (1/2/3; identity
// for TRK_AXIS_NONE) with sine s and cosine c.
__device__ __forceinline__ dfl rot_entry(int axis, dfl s, dfl c, int i, int j)
{
    const dfl one = df_from(1.0f), zero = df_from(0.0f);
    if (axis == TRK_AXIS_NONE) return i == j ? one : zero;
    const int a = axis - 1;  // the fixed coordinate
    if (i == a || j == a) return i == j ? one : zero;
    if (i == j) return c;
    // x: (1,2) = -s, (2,1) = s; y: (0,2) = s, (2,0) = -s; z: (0,1) = -s, (1,0) = s
    const bool neg = (axis == TRK_AXIS_Y) ? (i > j) : (i < j);
    return neg ? df_neg(s) : s;
}

// Projective rows of every frame for one instrument state, in double-float, by
// one warp or two (compose_joints and compose_pose side by side, a block barrier,
// compose_chain): rows (fx M0, fy M1, M2) of M = T_r^c T_f(q) with
// T_f = T_parent * [Rot(axis_f, coef_f q_joint) | offset_f] and q from the
// inverse cosine map q = lb + (ub-lb)/2 (1 - cos(pi (qh-lb)/(ub-lb))),
// written as hi/lo float pairs (24 floats per frame).  The pose rotation is
// axis-angle, R = cos t I + sin t [k]x + (1 - cos t) k k^T with t = |r|,
// k = r / t (I + [r]x when t < 1e-8), or look-at Ry(gamma) Rx(alpha) Rz(beta)
// (Sec. III-A.3).  The lanes run the same code on different data: one
// sine/cosine evaluation gives the three joint maps, a second one the joint
// rotations, a third one the pose, then the chain products, level by level
// (frames at the same distance from the root in parallel).  All of it is latency
// that the CTA waits for: 9.1k cycles with one warp and sine and cosine on every
// lane, 6.8k with two warps and a polynomial per lane (640x512, 64 candidates:
// 34.1 -> 32.9 us).  The chain's root starts from G = diag(fx, fy, 1) [R | t], so
// each product down the chain yields the frame's scaled projective rows directly.
// scr: kComposeScratch float2 (a multiple of two, so what follows stays
// 16-byte aligned).
constexpr int kComposeScratch = 4 + 12 + kMaxFrames * 9 + kMaxFrames * 12;

// The joint rotations (Js of the scratch): lanes 0-2 the joint maps, then lane f
// frame f's rotation.
static __device__ void compose_joints(const ChainDev &ch, const float *st, float2 *scr, int lane)
{
    float2 *qs = scr, *Js = scr + 16;
    const int nF = ch.n_frames;
    dfl arg = df_from(0.0f);
    if (lane < 3) arg = df_mul(df_sub(df_from(st[6 + lane]), dfc(ch.lb_df[lane])), dfc(ch.pi_over_range_df[lane]));
    const dfl2 sc = df_sincos16(arg);
    if (lane < 3) {
        const dfl q = df_fma(dfc(ch.half_range_df[lane]), df_sub(df_from(1.0f), sc.c), dfc(ch.lb_df[lane]));
        qs[lane] = make_float2(q.hi, q.lo);
    }
    __syncwarp();
    dfl ang = df_from(0.0f);
    if (lane < nF) ang = df_mul(dfc(ch.coef_df[lane]), dfc(qs[ch.joint[lane]]));
    const dfl2 fsc = df_sincos16(ang);
    if (lane < nF) {
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const dfl v = rot_entry(ch.axis[lane], fsc.s, fsc.c, e / 3, e % 3);
            Js[9 * lane + e] = make_float2(v.hi, v.lo);
        }
    }
}

// G of the scratch, from the pose angle t = |r| (lane 0) or the look-at angles
// gamma, alpha, beta (lanes 0-2); lanes 0-8 hold the rotation's entries.
static __device__ void compose_pose(const ChainDev &ch, const CamDev &cam, const float *st, float2 *scr, int lane)
{
    float2 *G = scr + 4, *Ts = scr + 16 + kMaxFrames * 9;
    const bool lookat = ch.rot_param == TRK_ROT_LOOKAT;
    const dfl r0 = df_from(st[0]), r1 = df_from(st[1]), r2 = df_from(st[2]);
    const dfl t = lookat ? df_from(0.0f) : df_sqrt(dot3(r0, r0, r1, r1, r2, r2));
    const dfl2 sc = df_sincos16(lookat ? (lane == 0 ? r2 : lane == 1 ? r0 : r1) : t);
    if (lane < 3) {  // sines and cosines, parked in the chain scratch
        Ts[2 * lane] = make_float2(sc.s.hi, sc.s.lo);
        Ts[2 * lane + 1] = make_float2(sc.c.hi, sc.c.lo);
    }
    __syncwarp();
    dfl Rv = df_from(0.0f);
    if (lane < 9) {
        const int i = lane / 3, j = lane - 3 * (lane / 3);
        if (lookat) {
            const dfl sg = dfc(Ts[0]), cg = dfc(Ts[1]), sa = dfc(Ts[2]), ca = dfc(Ts[3]), sb = dfc(Ts[4]),
                      cb = dfc(Ts[5]);
            dfl row[3];  // row i of Ry(gamma) Rx(alpha)
#pragma unroll
            for (int l = 0; l < 3; ++l)
                row[l] = dot3(rot_entry(TRK_AXIS_Y, sg, cg, i, 0), rot_entry(TRK_AXIS_X, sa, ca, 0, l),
                              rot_entry(TRK_AXIS_Y, sg, cg, i, 1), rot_entry(TRK_AXIS_X, sa, ca, 1, l),
                              rot_entry(TRK_AXIS_Y, sg, cg, i, 2), rot_entry(TRK_AXIS_X, sa, ca, 2, l));
            Rv = dot3(row[0], rot_entry(TRK_AXIS_Z, sb, cb, 0, j), row[1], rot_entry(TRK_AXIS_Z, sb, cb, 1, j),
                      row[2], rot_entry(TRK_AXIS_Z, sb, cb, 2, j));
        } else {
            const dfl r[3] = {r0, r1, r2};
            if (t.hi < 1e-8f) {
                // I + [r]x: (0,1) = -r2, (0,2) = r1, (1,0) = r2, (1,2) = -r0, (2,0) = -r1, (2,1) = r0
                const int m = 3 - i - j;
                const bool neg = ((i + 1) % 3) == j;
                Rv = i == j ? df_from(1.0f) : (neg ? df_neg(r[m]) : r[m]);
            } else {
                const dfl it = df_div(df_from(1.0f), t);
                const dfl s = dfc(Ts[0]), c = dfc(Ts[1]);
                const dfl ki = df_mul(r[i], it), kj = df_mul(r[j], it);
                dfl Kij = df_from(0.0f);
                if (i != j) {
                    const int m = 3 - i - j;
                    const bool neg = ((i + 1) % 3) == j;
                    const dfl km = df_mul(r[m], it);
                    Kij = neg ? df_neg(km) : km;
                }
                Rv = df_fma(df_sub(df_from(1.0f), c), df_mul(ki, kj), df_mul(s, Kij));
                if (i == j) Rv = df_add(Rv, c);
            }
        }
    }
    // G = diag(fx, fy, 1) [R | t], row-major 3 x 4: lanes 0-8 the rotation
    // entries, lanes 9-11 the translation
    if (lane < 12) {
        const int i = lane < 9 ? lane / 3 : lane - 9;
        dfl g = lane < 9 ? Rv : df_from(st[3 + i]);
        if (i == 0) g = df_mul(g, dfc(cam.fx_df));
        if (i == 1) g = df_mul(g, dfc(cam.fy_df));
        G[lane < 9 ? 4 * i + (lane - 3 * i) : 4 * i + 3] = make_float2(g.hi, g.lo);
    }
}

// The chain from G and the joint rotations to the frames' scaled rows.
static __device__ void compose_chain(const ChainDev &ch, float *out, float2 *scr, int lane)
{
    float2 *G = scr + 4, *Js = scr + 16, *Ts = scr + 16 + kMaxFrames * 9;
    const int nF = ch.n_frames;
    // the chain, level by level (a frame's level is its distance from the root):
    // the frames of one level are independent, two at a time (12 lanes each,
    // lane = 4 i + j within a frame)
    int lvl = 0;
    if (lane < nF)
        for (int q = ch.parent[lane]; q >= 0; q = ch.parent[q]) ++lvl;
    int top = lvl;
    for (int o = 16; o; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    for (int l = 0; l <= top; ++l) {
        for (unsigned fm = __ballot_sync(0xffffffffu, lane < nF && lvl == l); fm;) {
            const int fa = __ffs(fm) - 1;
            fm &= fm - 1;
            const int fb = fm ? __ffs(fm) - 1 : -1;
            if (fm) fm &= fm - 1;
            const int f = lane < 12 ? fa : (lane < 24 ? fb : -1);
            if (f >= 0) {
                const int e = lane < 12 ? lane : lane - 12, i = e >> 2, jj = e & 3;
                const float2 *Jf = Js + 9 * f;
                dfl L0 = jj < 3 ? dfc(Jf[jj]) : dfc(ch.offset_df[f][0]);
                dfl L1 = jj < 3 ? dfc(Jf[3 + jj]) : dfc(ch.offset_df[f][1]);
                dfl L2 = jj < 3 ? dfc(Jf[6 + jj]) : dfc(ch.offset_df[f][2]);
                const float2 *P = ch.parent[f] < 0 ? G : Ts + 12 * ch.parent[f];
                dfl v = dot3(dfc(P[4 * i]), L0, dfc(P[4 * i + 1]), L1, dfc(P[4 * i + 2]), L2);
                if (jj == 3) v = df_add(v, dfc(P[4 * i + 3]));
                Ts[12 * f + e] = make_float2(v.hi, v.lo);
            }
            __syncwarp();
        }
    }
    for (int e = lane; e < nF * 12; e += 32) {  // scaled rows of M_f, hi then lo
        const int f = e / 12, r = e - 12 * f;
        const float2 v = Ts[e];
        out[24 * f + r] = v.x;
        out[24 * f + 12 + r] = v.y;
    }
    __syncwarp();
}

// All of it by one warp.
static __device__ void compose_frames_warp(const ChainDev &ch, const CamDev &cam, const float *st, float *out,
                                           float2 *scr, int lane)
{
    compose_joints(ch, st, scr, lane);
    compose_pose(ch, cam, st, scr, lane);
    __syncwarp();
    compose_chain(ch, out, scr, lane);
}

// ----------------------------------------------------------------------------
// Compensated FP32 ("double-float") arithmetic: Knuth's TwoSum and the
// FMA-based TwoProd give exact rounding errors; explicit _rn intrinsics keep
// the compiler from contracting them.
// ----------------------------------------------------------------------------
struct DF {
    float hi, lo;
};

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e)
{
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// hi + lo renormalised, |hi| >= |lo| (Dekker's FastTwoSum)
__device__ __forceinline__ DF fast_two_sum(float hi, float lo)
{
    DF r;
    r.hi = __fadd_rn(hi, lo);
    r.lo = __fsub_rn(lo, __fsub_rn(r.hi, hi));
    return r;
}

// (hi + lo) . (x, y, z, 1).  The sum of the rounding errors is below the sum
// itself unless the row cancels to nothing, and then what FastTwoSum loses is
// below the errors' own rounding.
__device__ __forceinline__ DF df_affine(const float *h, const float *l, float x, float y, float z)
{
    float p0, e0, p1, e1, p2, e2, s, t0, t1, t2;
    two_prod(h[0], x, p0, e0);
    two_prod(h[1], y, p1, e1);
    two_prod(h[2], z, p2, e2);
    two_sum(p0, p1, s, t0);
    two_sum(s, p2, s, t1);
    two_sum(s, h[3], s, t2);
    float err = __fadd_rn(__fadd_rn(t0, t1), __fadd_rn(t2, e0));
    err = __fadd_rn(err, __fadd_rn(e1, e2));
    err = __fadd_rn(err, __fmaf_rn(l[0], x, __fmaf_rn(l[1], y, __fmaf_rn(l[2], z, l[3]))));
    return fast_two_sum(s, err);
}

// a / b given rb = 1/b.hi (approximate): one correction step from the residual
// (a.hi - q1 b.hi is exact: q1 is the quotient to within a few ulp).
__device__ __forceinline__ DF df_div(DF a, DF b, float rb)
{
    const float q1 = __fmul_rn(a.hi, rb);
    const float r = __fadd_rn(__fmaf_rn(-q1, b.hi, a.hi), __fmaf_rn(-q1, b.lo, a.lo));
    return fast_two_sum(q1, __fmul_rn(r, rb));
}

// Round-half-even of 256 (hi + lo), exact for |256 hi| <= 2^22 (the guard band):
// adding 1.5 2^23 rounds to an integer and leaves it in the low mantissa bits.
__device__ __forceinline__ int snap256(DF u)
{
    const float magic = 12582912.0f;  // 1.5 * 2^23
    const float a = __fmul_rn(u.hi, 256.0f);
    const float t = __fadd_rn(a, magic);
    int n = __float_as_int(t) - __float_as_int(magic);
    const float d = __fsub_rn(a, __fsub_rn(t, magic));
    if (fabsf(d) == 0.5f) {  // a tie of the high part: the low part decides
        if (d > 0.0f && u.lo > 0.0f) ++n;
        if (d < 0.0f && u.lo < 0.0f) --n;
    }
    return n;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ----------------------------------------------------------------------------
// Triangle setup shared by the raster paths.
// ----------------------------------------------------------------------------
struct TriSetup {
    int x[3], y[3];       // snapped vertices, positive orientation
    int j0, j1, i0, i1;   // pixel bbox clamped to the image
    int spanx, spany;     // vertex bbox extent in 1/256 px
};

// Returns 0 = nothing to draw, 1 = draw, 2 = culled for a flagged vertex.
// The clipped pixel bounding box is tested first: most triangles of a fine
// mesh contain no pixel centre and leave before the orientation test.
__device__ __forceinline__ int tri_setup(int2 a, int2 b, int2 c, int W, int H, int cull, TriSetup &t)
{
    if (a.x == kSnapFlag || b.x == kSnapFlag || c.x == kSnapFlag) return 2;
    int xmn = min(a.x, min(b.x, c.x)), xmx = max(a.x, max(b.x, c.x));
    int ymn = min(a.y, min(b.y, c.y)), ymx = max(a.y, max(b.y, c.y));
    t.j0 = max(0, (xmn + 255) >> 8);   // ceil(x / 256)
    t.j1 = min(W - 1, xmx >> 8);       // floor(x / 256)
    t.i0 = max(0, (ymn + 255) >> 8);
    t.i1 = min(H - 1, ymx >> 8);
    if (t.j0 > t.j1 || t.i0 > t.i1) return 0;
    t.spanx = xmx - xmn;
    t.spany = ymx - ymn;
    long long A;
    if (t.spanx < (1 << 15) && t.spany < (1 << 15)) {  // |products| < 2^30: int32 is exact
        A = (long long)((b.x - a.x) * (c.y - a.y) - (c.x - a.x) * (b.y - a.y));
    } else {
        A = (long long)(b.x - a.x) * (long long)(c.y - a.y) - (long long)(c.x - a.x) * (long long)(b.y - a.y);
    }
    if (A == 0) return 0;
    if (cull && A > 0) return 0;
    if (A < 0) {
        int2 tmp = b;
        b = c;
        c = tmp;
    }
    t.x[0] = a.x; t.y[0] = a.y;
    t.x[1] = b.x; t.y[1] = b.y;
    t.x[2] = c.x; t.y[2] = c.y;
    return 1;
}

// Edge k runs from vertex k to vertex k+1.  e_k(j, i) = dx (256 i - y_k)
// - dy (256 j - x_k) - bias_k, bias 0 on top-left edges (dy < 0, or dy == 0 and
// dx > 0) and 1 otherwise, so a pixel is covered iff every e_k >= 0.
__device__ __forceinline__ long long edge64(const TriSetup &t, int k, long long Px, long long Py)
{
    int k1 = (k == 2) ? 0 : k + 1;
    long long dx = t.x[k1] - t.x[k], dy = t.y[k1] - t.y[k];
    int bias = (dy < 0 || (dy == 0 && dx > 0)) ? 0 : 1;
    return dx * (Py - t.y[k]) - dy * (Px - t.x[k]) - bias;
}

// One thread, int32 incremental edges.  Requires spanx < 32 px and spany < 64 px
// so that |e| < 2^28 over the bbox (also at its corner, so the start values
// are exact in int32) and a row fits one 64-bit word window.  Each row
// collects its coverage most-significant-bit first (a funnel shift per
// pixel), then one bit reversal puts pixel j0 at bit 0.
// `row` points at the bitmap word holding pixel (t.i0, t.j0 & ~31); rows are
// `stride` words apart.
__device__ __forceinline__ void raster_small_at(const TriSetup &t, uint32_t *row, int stride)
{
    int r[3], cs[3], rs[3];
    const int Px = 256 * t.j0, Py = 256 * t.i0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int k1 = (k == 2) ? 0 : k + 1;
        const int dx = t.x[k1] - t.x[k], dy = t.y[k1] - t.y[k];
        const int bias = (dy < 0 || (dy == 0 && dx > 0)) ? 0 : 1;
        r[k] = dx * (Py - t.y[k]) - dy * (Px - t.x[k]) - bias;
        cs[k] = dy * 256;
        rs[k] = dx * 256;
    }
    const int jb = t.j0 & ~31;
    const int off = t.j0 - jb;
    const int nb = t.j1 - t.j0 + 1;  // 1..32
    const bool one_word = off + nb <= 32;
    for (int i = t.i0; i <= t.i1; ++i) {
        int a0 = r[0], a1 = r[1], a2 = r[2];
        uint32_t bits = 0u;
#pragma unroll 4
        for (int n = 0; n < nb; ++n) {
            bits = __funnelshift_l((uint32_t)(~(a0 | a1 | a2)), bits, 1);  // (bits << 1) | covered
            a0 -= cs[0];
            a1 -= cs[1];
            a2 -= cs[2];
        }
        if (bits) {
            const uint32_t rb = __brev(bits) >> (32 - nb);  // pixel j0 at bit 0
            if (one_word) {
                atomicOr(row, rb << off);
            } else {  // off >= 1 here
                const uint32_t lo = rb << off, hi = rb >> (32 - off);
                if (lo) atomicOr(row, lo);
                if (hi) atomicOr(row + 1, hi);
            }
        }
        r[0] += rs[0];
        r[1] += rs[1];
        r[2] += rs[2];
        row += stride;
    }
}

__device__ __forceinline__ void raster_small(const TriSetup &t, uint32_t *bm, int Wq)
{
    raster_small_at(t, bm + (size_t)t.i0 * Wq + ((t.j0 & ~31) >> 5), Wq);
}

// One whole warp per triangle: lane l tests pixel 32 w + l of word w, int64 edges.
static __device__ void raster_warp(const TriSetup &t, uint32_t *bm, int Wq, int lane)
{
    for (int i = t.i0; i <= t.i1; ++i) {
        long long Py = 256LL * i;
        for (int w = t.j0 >> 5; w <= (t.j1 >> 5); ++w) {
            int j = (w << 5) + lane;
            bool in = (j >= t.j0) && (j <= t.j1);
            if (in) {
                long long Px = 256LL * j;
                long long e = edge64(t, 0, Px, Py) | edge64(t, 1, Px, Py) | edge64(t, 2, Px, Py);
                in = e >= 0;
            }
            unsigned m = __ballot_sync(0xffffffffu, in);
            if (lane == 0 && m) atomicOr(bm + (size_t)i * Wq + w, m);
        }
    }
}

// ----------------------------------------------------------------------------
// Quadrilaterals: two mesh triangles T1 = (a, b, c) and T2 = (a, c, d) that share
// the edge a-c.  The top-left rule covers a pixel centre p exactly when the
// point p + (e, e^2), e -> 0+, lies strictly inside the triangle (for a
// non-horizontal edge the x shift decides the side, for a horizontal one the y
// shift).  That point never lies on the diagonal a-c, and when both triangles
// have the same orientation and (a, b, c, d) is strictly convex, the open
// quadrilateral minus the diagonal is the union of the two open triangles.  So
// the pixels of the quadrilateral under the same rule on its four edges are
// exactly the union of the two triangles' pixels: one set-up and one pass over
// one bounding box instead of two.  Anything else (a fold at a silhouette edge,
// a non-convex or degenerate pair, a flagged vertex) is drawn as two triangles.
// ----------------------------------------------------------------------------
// Twice the signed area of (p, q, r).
__device__ __forceinline__ long long orient2(int2 p, int2 q, int2 r)
{
    return (long long)(q.x - p.x) * (long long)(r.y - p.y) - (long long)(r.x - p.x) * (long long)(q.y - p.y);
}

// ----------------------------------------------------------------------------
// Small primitives (corners spanning less than 32 px across and 64 px down, so
// that int32 edge functions are exact over the box and its corner, and a row
// fits one 64-bit window) drawn a row per lane.
// ----------------------------------------------------------------------------

// A primitive's corners (c3.x == kSnapFlag: a triangle); part: which of its
// record's triangles it stands for (0 both, 1 the first, 2 the second).
struct PrimEntry {
    int2 c0, c1, c2, c3;
    int part;
};

// The entry of a record's snapped corners: triangles with a flagged corner are
// left out (and counted).  False: nothing left.
__device__ __forceinline__ bool make_entry(int2 v0, int2 v1, int2 v2, int2 v3, bool pair, int &culled, PrimEntry &e)
{
    const bool f = v0.x == kSnapFlag || v2.x == kSnapFlag;
    const bool fa = f || v1.x == kSnapFlag, fb = pair && (f || v3.x == kSnapFlag);
    culled += fa + fb;
    e.c0 = v0;
    e.c1 = v1;
    e.c2 = v2;
    e.c3 = v3;
    e.part = pair ? 0 : 1;
    if (!pair || fb) {
        e.c3.x = kSnapFlag;
        e.part = 1;
        return !fa;
    }
    if (fa) {
        e.c1 = v2;
        e.c2 = v3;
        e.c3.x = kSnapFlag;
        e.part = 2;
    }
    return true;
}

// Pixel box of an entry, clipped to the image.  Returns 0: no pixel centre in
// it, 1: small, 2: large.
__device__ __forceinline__ int entry_size(const PrimEntry &e, int W, int H)
{
    const int2 c3 = e.c3.x == kSnapFlag ? e.c2 : e.c3;
    const int xmn = min(min(e.c0.x, e.c1.x), min(e.c2.x, c3.x)), xmx = max(max(e.c0.x, e.c1.x), max(e.c2.x, c3.x));
    const int ymn = min(min(e.c0.y, e.c1.y), min(e.c2.y, c3.y)), ymx = max(max(e.c0.y, e.c1.y), max(e.c2.y, c3.y));
    if (max(0, (xmn + 255) >> 8) > min(W - 1, xmx >> 8) || max(0, (ymn + 255) >> 8) > min(H - 1, ymx >> 8)) return 0;
    return xmx - xmn < 32 * 256 && ymx - ymn < 64 * 256 ? 1 : 2;
}

__device__ __forceinline__ int orient_small(int2 p, int2 q, int2 r)
{
    return (q.x - p.x) * (r.y - p.y) - (r.x - p.x) * (q.y - p.y);
}

// No triangle of a small entry faces the camera (negative orientation).
__device__ __forceinline__ bool back_small(const PrimEntry &e)
{
    return orient_small(e.c0, e.c1, e.c2) >= 0 && (e.c3.x == kSnapFlag || orient_small(e.c0, e.c2, e.c3) >= 0);
}

// A warp draws the small primitives that its lanes hold (`live`), a row of
// pixels per lane: rows, not primitives, are shared out, so the lanes work alike
// whatever the primitives' sizes.  A pair of triangles is drawn as one convex
// quadrilateral where it is one, else as its triangles, one after the other;
// `cull` leaves out the back faces.  tab: the warp's table of n entries, n at
// least the number of live lanes: the polygons' edge functions at the first
// pixel of their box (int4 [n]), edge vectors (int4 [n], dx and dy in 16 bits),
// first task, columns and place in the bitmap (int2 [n]).
__device__ __forceinline__ void draw_rows(bool live, int2 c0, int2 c1, int2 c2, int2 c3, int W, int H, int cull,
                                          uint32_t *bm, int Wq, int4 *tab, int n, int lane)
{
    int4 *tab_r = tab, *tab_d = tab + n;
    int2 *tab_m = reinterpret_cast<int2 *>(tab + 2 * n);
    bool tri = c3.x == kSnapFlag, two = false;
    const int2 mid = c2, end = c3;
    int A = 0;
    if (live) {
        A = orient_small(c0, c1, c2);
        if (!tri) {
            const int A2 = orient_small(c0, c2, c3);
            const int Da = orient_small(c1, c3, c0), Dc = orient_small(c1, c3, c2);
            // same non-zero orientation, and c0, c2 strictly on opposite sides of c1-c3
            if (!(((A > 0 && A2 > 0) || (A < 0 && A2 < 0)) && ((Da > 0 && Dc < 0) || (Da < 0 && Dc > 0)))) tri = two = true;
        }
    }
    for (;;) {
        bool on = live && A != 0 && !(cull && A > 0);
        int4 r, d;
        int2 m;
        int rows = 0;
        if (on) {
            if (A < 0) {  // positive orientation
                const int2 t = c1;
                c1 = tri ? c2 : c3;
                (tri ? c2 : c3) = t;
            }
            if (tri) c3 = c2;
            const int j0 = max(0, (min(min(c0.x, c1.x), min(c2.x, c3.x)) + 255) >> 8);
            const int j1 = min(W - 1, max(max(c0.x, c1.x), max(c2.x, c3.x)) >> 8);
            const int i0 = max(0, (min(min(c0.y, c1.y), min(c2.y, c3.y)) + 255) >> 8);
            const int i1 = min(H - 1, max(max(c0.y, c1.y), max(c2.y, c3.y)) >> 8);
            on = j0 <= j1 && i0 <= i1;
            rows = on ? i1 - i0 + 1 : 0;
            const int Px = 256 * j0, Py = 256 * i0;
            auto edge = [&](int2 p, int2 q, int &rv, int &dv) {
                const int dx = q.x - p.x, dy = q.y - p.y;
                const int bias = (dy < 0 || (dy == 0 && dx > 0)) ? 0 : 1;
                rv = dx * (Py - p.y) - dy * (Px - p.x) - bias;
                dv = (int)((unsigned)dx << 16 | ((unsigned)dy & 0xffffu));
            };
            edge(c0, c1, r.x, d.x);
            edge(c1, c2, r.y, d.y);
            edge(c2, c3, r.z, d.z);
            edge(c3, c0, r.w, d.w);
            if (tri) r.z = 0;  // the edge from c2 to c2: no constraint (its steps are 0)
            m.x = (j1 - j0) << 16 | (j0 & 31) << 24;
            m.y = i0 * Wq + (j0 >> 5);
        }
        int incl = rows;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31), first = incl - rows;
        const unsigned lm = __ballot_sync(0xffffffffu, on);
        if (on) {
            const int slot = __popc(lm & ((1u << lane) - 1u));
            m.x |= first;
            tab_r[slot] = r;
            tab_d[slot] = d;
            tab_m[slot] = m;
        }
        __syncwarp();
        for (int base = 0; base < total; base += 32) {
            // the polygon of task base + lane: those that start before this
            // window, then one more at each start within it
            const int rel = first - base;
            const unsigned starts = __reduce_or_sync(0xffffffffu, on && rel >= 0 && rel < 32 ? 1u << rel : 0u);
            const int before = __popc(__ballot_sync(0xffffffffu, on && rel < 0));
            const int t = base + lane;
            if (t < total) {
                const int slot = before - 1 + __popc(starts & (0xffffffffu >> (31 - lane)));
                const int4 rv = tab_r[slot], dv = tab_d[slot];
                const int2 mv = tab_m[slot];
                const int row = t - (mv.x & 0xffff), nb = (mv.x >> 16 & 31) + 1, off = mv.x >> 24;
                const int cs0 = (int)((unsigned)dv.x << 16) >> 8, cs1 = (int)((unsigned)dv.y << 16) >> 8;  // 256 dy
                const int cs2 = (int)((unsigned)dv.z << 16) >> 8, cs3 = (int)((unsigned)dv.w << 16) >> 8;
                int a0 = rv.x + row * 256 * (dv.x >> 16), a1 = rv.y + row * 256 * (dv.y >> 16);
                int a2 = rv.z + row * 256 * (dv.z >> 16), a3 = rv.w + row * 256 * (dv.w >> 16);
                uint32_t bits = 0u;
#pragma unroll 4
                for (int q = 0; q < nb; ++q) {
                    bits = __funnelshift_l((uint32_t)(~(a0 | a1 | a2 | a3)), bits, 1);  // (bits << 1) | covered
                    a0 -= cs0;
                    a1 -= cs1;
                    a2 -= cs2;
                    a3 -= cs3;
                }
                if (bits) {
                    const uint32_t rb = __brev(bits) >> (32 - nb);  // pixel j0 at bit 0
                    uint32_t *w = bm + mv.y + row * Wq;
                    const uint32_t lo = rb << off, hi = off ? rb >> (32 - off) : 0u;
                    if (lo) atomicOr(w, lo);
                    if (hi) atomicOr(w + 1, hi);
                }
            }
        }
        __syncwarp();
        if (!__any_sync(0xffffffffu, two)) break;
        live = two;  // the second triangles
        two = false;
        tri = true;
        if (live) {
            c1 = mid;
            c2 = end;
            A = orient_small(c0, c1, c2);
        }
    }
}

// floor(n / d) for 0 < d < 2^24, clamped to [-cap - 2, cap + 1] (cap < 2^21): a
// quotient in FP32, once clamped within one of the floor, is put right by its
// exact remainder.
__device__ __forceinline__ int floor_div_clamped(long long n, int d, int cap)
{
    const float f = fminf(fmaxf((float)n * rcp_approx((float)d), (float)(-cap - 1)), (float)cap);
    int q = (int)floorf(f);
    const long long r = n - (long long)q * d;
    if (r < 0) --q;
    if (r >= d) ++q;
    return q;
}

// The columns [lo, hi] of row i that the edge p -> q leaves covered (e >= 0, see
// edge64): one floor of the edge function over its step.  An edge of no length
// leaves all.
__device__ __forceinline__ void clip_row(int2 p, int2 q, int i, int &lo, int &hi)
{
    const int dx = q.x - p.x, dy = q.y - p.y;
    const int bias = (dy < 0 || (dy == 0 && dx > 0)) ? 0 : 1;
    // e at column lo; e falls by 256 dy per column
    const long long e = (long long)dx * (256 * i - p.y) - (long long)dy * (256 * lo - p.x) - bias;
    if (dy == 0) {
        if (dx != 0 && e < 0) hi = lo - 1;
        return;
    }
    const int n = hi - lo + 1, f = floor_div_clamped(e >> 8, abs(dy), max(n, 0));
    if (dy > 0) hi = min(hi, lo + f);      // columns up to lo + floor(e / 256 dy)
    else lo = max(lo, lo - f);             // from lo + ceil(-e / 256 |dy|)
}

// draw_rows for primitives of any size: a row of pixels per lane again, but the
// row's covered columns come from the edges (a convex polygon covers one run of
// them) and are entered a word at a time.  The entries of the warp's table are
// the corners (int4 [n] twice) and the first task and row (int2 [n]).
// 1280x1024, two instruments of 40k triangles, 256 candidates: with a pixel per
// lane and 64-bit edge functions at each, this phase took 76-160k cycles of the
// kernel's 160-250k, now 8-11k of 90-100k (1.90 -> 1.03 ms a launch).
static __device__ void draw_rows_large(bool live, int2 c0, int2 c1, int2 c2, int2 c3, int W, int H, int cull, uint32_t *bm,
                                       int Wq, int4 *tab, int n, int lane)
{
    int4 *tab_a = tab, *tab_b = tab + n;
    int2 *tab_m = reinterpret_cast<int2 *>(tab + 2 * n);
    bool tri = c3.x == kSnapFlag, two = false;
    const int2 mid = c2, end = c3;
    long long A = 0;
    if (live) {
        A = orient2(c0, c1, c2);
        if (!tri) {
            const long long A2 = orient2(c0, c2, c3), Da = orient2(c1, c3, c0), Dc = orient2(c1, c3, c2);
            // same non-zero orientation, and c0, c2 strictly on opposite sides of c1-c3
            if (!(((A > 0 && A2 > 0) || (A < 0 && A2 < 0)) && ((Da > 0 && Dc < 0) || (Da < 0 && Dc > 0)))) tri = two = true;
        }
    }
    for (;;) {
        bool on = live && A != 0 && !(cull && A > 0);
        int i0 = 0, rows = 0;
        if (on) {
            if (A < 0) {  // positive orientation
                const int2 t = c1;
                c1 = tri ? c2 : c3;
                (tri ? c2 : c3) = t;
            }
            if (tri) c3 = c2;
            i0 = max(0, (min(min(c0.y, c1.y), min(c2.y, c3.y)) + 255) >> 8);
            const int i1 = min(H - 1, max(max(c0.y, c1.y), max(c2.y, c3.y)) >> 8);
            on = i0 <= i1;
            rows = on ? i1 - i0 + 1 : 0;
        }
        int incl = rows;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31), first = incl - rows;
        const unsigned lm = __ballot_sync(0xffffffffu, on);
        if (on) {
            const int slot = __popc(lm & ((1u << lane) - 1u));
            tab_a[slot] = make_int4(c0.x, c0.y, c1.x, c1.y);
            tab_b[slot] = make_int4(c2.x, c2.y, c3.x, c3.y);
            tab_m[slot] = make_int2(first, i0);
        }
        __syncwarp();
        for (int base = 0; base < total; base += 32) {
            // the polygon of task base + lane, as in draw_rows
            const int rel = first - base;
            const unsigned starts = __reduce_or_sync(0xffffffffu, on && rel >= 0 && rel < 32 ? 1u << rel : 0u);
            const int before = __popc(__ballot_sync(0xffffffffu, on && rel < 0));
            const int t = base + lane;
            if (t < total) {
                const int slot = before - 1 + __popc(starts & (0xffffffffu >> (31 - lane)));
                const int4 pa = tab_a[slot], pb = tab_b[slot];
                const int2 mv = tab_m[slot];
                const int i = t - mv.x + mv.y;
                int lo = max(0, (min(min(pa.x, pa.z), min(pb.x, pb.z)) + 255) >> 8);
                int hi = min(W - 1, max(max(pa.x, pa.z), max(pb.x, pb.z)) >> 8);
                clip_row(make_int2(pa.x, pa.y), make_int2(pa.z, pa.w), i, lo, hi);
                clip_row(make_int2(pa.z, pa.w), make_int2(pb.x, pb.y), i, lo, hi);
                clip_row(make_int2(pb.x, pb.y), make_int2(pb.z, pb.w), i, lo, hi);
                clip_row(make_int2(pb.z, pb.w), make_int2(pa.x, pa.y), i, lo, hi);
                if (lo <= hi) {
                    uint32_t *w = bm + i * Wq;
                    for (int k = lo >> 5; k <= hi >> 5; ++k) {
                        uint32_t bits = 0xffffffffu;
                        if (k == lo >> 5) bits &= 0xffffffffu << (lo & 31);
                        if (k == hi >> 5) bits &= 0xffffffffu >> (31 - (hi & 31));
                        atomicOr(w + k, bits);
                    }
                }
            }
        }
        __syncwarp();
        if (!__any_sync(0xffffffffu, two)) break;
        live = two;  // the second triangles
        two = false;
        tri = true;
        if (live) {
            c1 = mid;
            c2 = end;
            A = orient2(c0, c1, c2);
        }
    }
}

// Camera-frame position of one vertex from its frame's projective rows (hi/lo
// pairs), perspective division and snap: int2 (U, V) in 1/256 px, or the flag
// value when the vertex is behind z_near or outside the guard band; uv gets
// the unsnapped offsets from the principal point.
__device__ __forceinline__ int2 project_vertex(float4 p, const float *Mh, const CamDev &cam, float2 &uv)
{
    DF X = df_affine(Mh + 0, Mh + 12, p.x, p.y, p.z);
    DF Y = df_affine(Mh + 4, Mh + 16, p.x, p.y, p.z);
    DF Z = df_affine(Mh + 8, Mh + 20, p.x, p.y, p.z);
    int2 o = make_int2(kSnapFlag, kSnapFlag);
    uv = make_float2(0.f, 0.f);
    if (Z.hi >= (float)cam.z_near) {
        const float rz = rcp_approx(Z.hi);
        DF u = df_div(X, Z, rz), w = df_div(Y, Z, rz);
        uv = make_float2(__fadd_rn(u.hi, u.lo), __fadd_rn(w.hi, w.lo));
        const float guard = (float)cam.guard;
        if (fabsf(u.hi) <= guard && fabsf(w.hi) <= guard)
            o = make_int2(snap256(u) + cam.cx256, snap256(w) + cam.cy256);
    }
    return o;
}

// ----------------------------------------------------------------------------
// Keypoint term (Eq. kpts_loss): the two keypoints of each instrument (the jaw
// tips) projected with the candidate's frames, compared with the detections
// under the better of the two assignments, plus their means, each distance
// reduced by the threshold tau and clipped at zero; summed over the
// instruments whose detection is valid (exactly two keypoints found), times
// lambda_kpts.  FP32 from the double-float frame rows.
// ----------------------------------------------------------------------------
__device__ __forceinline__ float2 project_keypoint(const float *M, const float *pt, const CamDev &cam)
{
    // rows (fx M0, fy M1, M2) as hi/lo pairs: M[r] hi, M[12 + r] lo, r = 4 i + j
    float X[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float acc = M[4 * i + 3] + M[12 + 4 * i + 3];
#pragma unroll
        for (int j = 0; j < 3; ++j) acc = fmaf(M[4 * i + j] + M[12 + 4 * i + j], pt[j], acc);
        X[i] = acc;
    }
    return make_float2(X[0] / X[2] + cam.cx256 * (1.0f / 256.0f), X[1] / X[2] + cam.cy256 * (1.0f / 256.0f));
}

__device__ __forceinline__ float pos_part(float x) { return fmaxf(x, 0.0f); }

static __device__ float keypoint_loss(const EvalArgs &a, const float *sM)
{
    const int nF = a.ch.n_frames;
    float total = 0.0f;
    for (int b = 0; b < a.ch.n_inst; ++b) {
        const float *o = a.kp_obs + 5 * b;
        if (o[4] == 0.0f) continue;
        const float2 p0 = project_keypoint(sM + (b * nF + a.kp_frame[0]) * 24, a.kp_pt[0], a.cam);
        const float2 p1 = project_keypoint(sM + (b * nF + a.kp_frame[1]) * 24, a.kp_pt[1], a.cam);
        const float tau = a.kp_tau;
        const float same = pos_part(hypotf(o[0] - p0.x, o[1] - p0.y) - tau) + pos_part(hypotf(o[2] - p1.x, o[3] - p1.y) - tau);
        const float swap = pos_part(hypotf(o[0] - p1.x, o[1] - p1.y) - tau) + pos_part(hypotf(o[2] - p0.x, o[3] - p0.y) - tau);
        const float mean = pos_part(hypotf(0.5f * (o[0] + o[2]) - 0.5f * (p0.x + p1.x), 0.5f * (o[1] + o[3]) - 0.5f * (p0.y + p1.y)) - tau);
        total += fminf(same, swap) + mean;
    }
    return a.kp_lambda * total;
}

// A candidate's state with a NaN or an infinity: its projection flags every
// vertex; report it in the device error word (one warp per CTA calls this).
__device__ __forceinline__ void check_state_finite(const float *st, int d, unsigned *err, int lane)
{
    const bool bad = lane < d && !isfinite(st[lane]);
    if (__ballot_sync(0xffffffffu, bad) && lane == 0 && err) atomicOr(err, TRK_DEVERR_NONFINITE);
}

// Programmatic dependent launch: kernels that follow each other on a stream
// are launched with programmatic stream serialisation, so the next kernel's
// CTAs may be scheduled while this one is still running; they wait for this
// grid to complete, memory included, before reading anything it writes.
// Without that launch attribute both instructions do nothing.
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace trk
