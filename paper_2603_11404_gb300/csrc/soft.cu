// Soft (differentiable) silhouette loss and its gradient: soft_eval and
// soft_refine in include/tracker.h.
//
// The soft form of the fitness (the paper fits with a differentiable
// renderer, Sec. III-A.2, and the MSE term of Eq. render_loss):
//   d_t(p)  signed distance (px) from pixel centre p to the boundary of
//           projected triangle t (+ inside, - outside), unsnapped coordinates
//   a_t(p)  sigmoid(d_t(p) / sigma), 0 where d_t(p) < -14 sigma
//   S(p)    1 - prod_t (1 - a_t(p)) = 1 - 1 / prod_t (1 + exp(d_t(p) / sigma))
//   L       sum_p (S(p) - M(p))^2
// and dL/dd_t(p) = 2 (S - M) (1 - S) sigmoid(d_t / sigma) / sigma, taken back
// through the closest boundary point to the projected vertices, through the
// pinhole to camera coordinates and through the kinematics to the state.
// Everything is FP32.
//
// Launches per call (one row of kernels per population):
//   k_soft_fk       per (candidate, instrument): kinematics with the nine
//                   state tangents carried along (forward mode); clears the
//                   candidate's accumulators
//   k_soft_tris     a warp per group of 32 triangles: projection, edge
//                   records, boxes; counts the groups that can reach each
//                   8x4-pixel block
//   k_soft_list     the blocks within reach, heavy ones first
//   k_soft_fwd      per listed block: the product over the triangles, the
//                   block's squared error and, for a gradient, the factor
//                   2 (S - M) (1 - S) / sigma of its pixels
//   k_soft_bwd      per pair of listed blocks: dL/d(u, v) of the triangles in
//                   reach over the blocks' pixels, added to the vertices
//   k_soft_reduce   dL/dX per vertex, reduced per kinematic frame to a 3x4
//                   matrix G_f, contracted with the tangents dT_f/dtheta_k
//
// Both pair kernels put triangles on the lanes and walk the pixels together:
// a triangle's record stays in registers (no shared-memory read per pair), the
// two coordinates of a pixel in an edge's frame are one FMA each from the
// previous ones, and nothing is exchanged between lanes per pair -- the forward
// keeps one running product per pixel and lane, the backward one sum per
// vertex coordinate and lane.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"

namespace trk {

constexpr float kSoftCutoff = 14.0f;   // in units of sigma
constexpr int kBlkW = 8, kBlkH = 4;    // pixel block of the pair kernels: one pixel per lane at its ends
constexpr int kBlkPx = kBlkW * kBlkH;
constexpr int kSoftThreads = 256;
constexpr int kFwdWarps = 4;           // warps that share a heavy block of the forward
constexpr int kBwdWarps = 4;           // and of the backward
// Groups within reach that make a block heavy.  On a small image there are too few
// blocks to hide one warp's long block behind the others: at 12, 8 candidates at
// 200x150 (loss and gradient, three scenes) take 329, 210 and 206 us, at 48 447, 243
// and 267; 64 at 101x77 513, 352 and 421 against 661, 471 and 484.  At 640x512 sharing
// costs more than it gives (64 candidates: 4.66, 2.24 and 2.42 ms against 4.29, 1.66
// and 1.95).  A rule on the image alone: a candidate's bits do not depend on the
// population it is called with.
constexpr int kHeavy = 48, kHeavySmall = 12, kSmallBlocks = 1024;
// With 1 + Q = prod (1 + exp): Q above kOne makes 1 - S < 2^-25, S is 1 in FP32
// and the pixel's gradient factor 0, whatever the remaining triangles add.  The
// forward stops early only at the larger kSaturated, so that a product formed
// in another order cannot fall below kOne again.
constexpr float kOne = 3.4e7f, kSaturated = 6.6e7f;
// A product over no triangle: nothing beside the smallest term (8e-7), and not
// zero, so that Q fma'd with an infinite product gives infinity, never NaN.
constexpr float kEmpty = 1e-30f;
// Gradient sums are accumulated in 64-bit fixed point, exact and so independent
// of the order of the (atomic) additions: dL/d(u, v) per vertex in units of
// 2^-36 (|sum| < 2^27: with x_t = softplus(d_t / sigma) >= sigmoid, a pixel adds
// at most 2 / sigma * sum_t sigmoid_t * exp(-sum_t x_t) <= 2 / (e sigma), so an
// image of TRK_MAX_PIXELS at the smallest sigma, 0.05 px, stays below 2^25),
// the per-frame G_f in units of 2^-24 (|sum| < 2^39) and the remainders in units
// of 2^-56 (a gradient that nearly vanishes keeps its digits).
constexpr float kGvScale = 68719476736.0f;
constexpr float kRestScale = 4294967296.0f;
constexpr float kGScale = 16777216.0f;
// The loss in units of 2^-41 (TRK_MAX_PIXELS of them stay below 2^62) and the
// blocks' remainders in units of 2^-73: an instrument that reaches into the image
// by its fringe alone has a loss of 1e-6 and less.
constexpr int kLossBits = 41;
constexpr float kLossScale = 2199023255552.0f;
// (a power of two times a float is exact in FP32: no FP64 arithmetic needed)
__device__ __forceinline__ long long to_fixed(float x, float scale) { return __float2ll_rn(x * scale); }

// ---------------------------------------------------------------------------
// Forward-mode kinematics: every lane carries the values and one tangent
// direction (lane k+1: d/dtheta_k, lane 0: none).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mul34(const float *A, const float *B, float *C)  // [R|t] * [R|t]
{
    float T[12];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float acc = (j == 3) ? A[4 * i + 3] : 0.0f;
#pragma unroll
            for (int k = 0; k < 3; ++k) acc = fmaf(A[4 * i + k], B[4 * k + j], acc);
            T[4 * i + j] = acc;
        }
#pragma unroll
    for (int e = 0; e < 12; ++e) C[e] = T[e];
}

// Derivative of the product C = A B of two [R|t] transforms:
// dC_R = dA_R B_R + A_R dB_R, dC_t = dA_R B_t + A_R dB_t + dA_t.
__device__ __forceinline__ void dmul34(const float *dA, const float *B, const float *A, const float *dB, float *dC)
{
    float T[12];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float acc = (j == 3) ? dA[4 * i + 3] : 0.0f;
#pragma unroll
            for (int k = 0; k < 3; ++k) acc = fmaf(dA[4 * i + k], B[4 * k + j], fmaf(A[4 * i + k], dB[4 * k + j], acc));
            T[4 * i + j] = acc;
        }
#pragma unroll
    for (int e = 0; e < 12; ++e) dC[e] = T[e];
}

// Elementary rotation about axis 1/2/3 (x/y/z) and its derivative by the angle.
__device__ __forceinline__ void rot_axis(int axis, float ang, float *R, float *dR)
{
    float s, c;
    sincosf(ang, &s, &c);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        R[e] = (e % 4 == 0) ? 1.0f : 0.0f;
        dR[e] = 0.0f;
    }
    if (axis == 1) {
        R[4] = c; R[5] = -s; R[7] = s; R[8] = c;
        dR[4] = -s; dR[5] = -c; dR[7] = c; dR[8] = -s;
    } else if (axis == 2) {
        R[0] = c; R[2] = s; R[6] = -s; R[8] = c;
        dR[0] = -s; dR[2] = c; dR[6] = -c; dR[8] = -s;
    } else if (axis == 3) {
        R[0] = c; R[1] = -s; R[3] = s; R[4] = c;
        dR[0] = -s; dR[1] = -c; dR[3] = c; dR[4] = -s;
    }
}

__device__ __forceinline__ void mul33(const float *A, const float *B, float *C)
{
    float T[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float acc = 0.0f;
#pragma unroll
            for (int k = 0; k < 3; ++k) acc = fmaf(A[3 * i + k], B[3 * k + j], acc);
            T[3 * i + j] = acc;
        }
#pragma unroll
    for (int e = 0; e < 9; ++e) C[e] = T[e];
}

// Rotation of the state and its derivative along r_dir (dir < 0: none).
// Axis-angle: Rodrigues R = I + s K + c1 K^2 (t = |r|, k = r / t, s = sin t,
// c1 = 1 - cos t, K = [k]x), differentiated term by term; below t = 1e-4 the
// second-order series I + [r]x + [r]x^2 / 2.  Look-at: Ry(g) Rx(a) Rz(b).
__device__ void rotation_tangent(int rot_param, const float r[3], int dir, float *R, float *dR)
{
    if (rot_param == TRK_ROT_LOOKAT) {
        float Ry[9], dRy[9], Rx[9], dRx[9], Rz[9], dRz[9], T[9];
        rot_axis(2, r[2], Ry, dRy);
        rot_axis(1, r[0], Rx, dRx);
        rot_axis(3, r[1], Rz, dRz);
        mul33(Ry, Rx, T);
        mul33(T, Rz, R);
        if (dir == 0) { mul33(Ry, dRx, T); mul33(T, Rz, dR); }
        else if (dir == 1) { mul33(Ry, Rx, T); mul33(T, dRz, dR); }
        else if (dir == 2) { mul33(dRy, Rx, T); mul33(T, Rz, dR); }
        else for (int e = 0; e < 9; ++e) dR[e] = 0.0f;
        return;
    }
    const float e0 = dir == 0 ? 1.0f : 0.0f, e1 = dir == 1 ? 1.0f : 0.0f, e2 = dir == 2 ? 1.0f : 0.0f;
    const float t = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
    if (t < 1e-4f) {
        // R = I + X + X^2 / 2 with X = [r]x; dR = E + (E X + X E) / 2, E = [e_dir]x
        float X[9] = {0, -r[2], r[1], r[2], 0, -r[0], -r[1], r[0], 0};
        float E[9] = {0, -e2, e1, e2, 0, -e0, -e1, e0, 0};
        float X2[9], EX[9], XE[9];
        mul33(X, X, X2);
        mul33(E, X, EX);
        mul33(X, E, XE);
        for (int e = 0; e < 9; ++e) {
            R[e] = ((e % 4 == 0) ? 1.0f : 0.0f) + X[e] + 0.5f * X2[e];
            dR[e] = E[e] + 0.5f * (EX[e] + XE[e]);
        }
        return;
    }
    const float it = 1.0f / t;
    const float k[3] = {r[0] * it, r[1] * it, r[2] * it};
    const float dt = (r[0] * e0 + r[1] * e1 + r[2] * e2) * it;  // d|r|
    const float dk[3] = {(e0 - k[0] * dt) * it, (e1 - k[1] * dt) * it, (e2 - k[2] * dt) * it};
    float s, c;
    sincosf(t, &s, &c);
    const float sh = sinf(0.5f * t);
    const float c1 = 2.0f * sh * sh, ds = c * dt, dc1 = s * dt;  // 1 - cos t without cancellation
    float K[9] = {0, -k[2], k[1], k[2], 0, -k[0], -k[1], k[0], 0};
    float dK[9] = {0, -dk[2], dk[1], dk[2], 0, -dk[0], -dk[1], dk[0], 0};
    float K2[9], A[9], B[9];
    mul33(K, K, K2);
    mul33(dK, K, A);
    mul33(K, dK, B);
    for (int e = 0; e < 9; ++e) {
        R[e] = ((e % 4 == 0) ? 1.0f : 0.0f) + s * K[e] + c1 * K2[e];
        dR[e] = ds * K[e] + s * dK[e] + dc1 * K2[e] + c1 * (A[e] + B[e]);
    }
}

// Camera-from-frame transforms of one instrument and their tangents along
// state direction `dir` (-1: none): T_f = T_c * T_E,f(q) (Sec. III-A.2).
__device__ void fk_tangent(const ChainDev &ch, const float *st, int dir, float (*T)[12], float (*dT)[12])
{
    float q[3], dq[3];
    for (int j = 0; j < 3; ++j) {
        const float lb = (float)ch.q_lb[j], ub = (float)ch.q_ub[j];
        if (ub == lb) {
            q[j] = lb;
            dq[j] = 0.0f;
        } else {
            const float a = 3.14159265358979f * (st[6 + j] - lb) / (ub - lb);
            float s, c;
            sincosf(a, &s, &c);
            q[j] = lb + 0.5f * (ub - lb) * (1.0f - c);       // Sec. III-A.3 inverse map
            dq[j] = (dir == 6 + j) ? 1.5707963267949f * s : 0.0f;  // d q / d qhat
        }
    }
    float R[9], dR[9];
    rotation_tangent(ch.rot_param, st, dir >= 0 && dir < 3 ? dir : -1, R, dR);
    float Tc[12] = {R[0], R[1], R[2], st[3], R[3], R[4], R[5], st[4], R[6], R[7], R[8], st[5]};
    const float dTc[12] = {dR[0], dR[1], dR[2], dir == 3 ? 1.0f : 0.0f, dR[3], dR[4], dR[5], dir == 4 ? 1.0f : 0.0f,
                           dR[6], dR[7], dR[8], dir == 5 ? 1.0f : 0.0f};
    float Tf[kMaxFrames][12], dTf[kMaxFrames][12];
    for (int f = 0; f < ch.n_frames; ++f) {
        float J[9], dJ[9];
        const float cf = (float)ch.coef[f];
        rot_axis(ch.axis[f], cf * q[ch.joint[f]], J, dJ);
        const float dang = cf * dq[ch.joint[f]];
        float L[12] = {J[0], J[1], J[2], (float)ch.offset[f][0], J[3], J[4], J[5], (float)ch.offset[f][1],
                       J[6], J[7], J[8], (float)ch.offset[f][2]};
        float dL[12] = {dJ[0] * dang, dJ[1] * dang, dJ[2] * dang, 0.0f, dJ[3] * dang, dJ[4] * dang, dJ[5] * dang,
                        0.0f, dJ[6] * dang, dJ[7] * dang, dJ[8] * dang, 0.0f};
        if (ch.axis[f] == 0)
            for (int e = 0; e < 12; ++e) dL[e] = 0.0f;
        const int p = ch.parent[f];
        if (p < 0) {
            for (int e = 0; e < 12; ++e) {
                Tf[f][e] = L[e];
                dTf[f][e] = dL[e];
            }
        } else {
            mul34(Tf[p], L, Tf[f]);
            dmul34(dTf[p], L, Tf[p], dL, dTf[f]);
        }
    }
    for (int f = 0; f < ch.n_frames; ++f) {
        mul34(Tc, Tf[f], T[f]);
        dmul34(dTc, Tf[f], Tc, dTf[f], dT[f]);
    }
}

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------
struct SoftArgs {
    ChainDev ch;
    int nF, nI, V, T, d, lam;
    float fx, fy, cx, cy, z_near, guard, sigma;
    int W, H, Wq;
    int nbx, nby;             // pixel blocks per row and column
    int heavy;                // groups within reach that make a block heavy
    int ngroups, NTp;         // groups of 32 triangles (over all instruments), triangles padded to whole groups
    int nsup;                 // runs of 32 groups
    const float4 *verts;
    const int4 *tris;
    const float *params;      // [lam * d]
    const uint32_t *mask;
    float *Tf;                // [lam * nI * nF * 12] camera-from-frame transforms
    float *dT;                // [lam * nI * nF * 9 * 12]
    float4 *rec;              // [4][lam * NTp] edge records (struct TriRec)
    float4 *box;              // [lam * NTp] centre and half extents of the triangle's bounding box
    short4 *gwin;             // [lam * ngroups] blocks that the group can reach: bx0, by0, bx1, by1 (bx0 > bx1: none)
    int4 *swin;               // [lam * nsup] the same for runs of 32 groups
    int *count;               // [lam * nby * nbx] groups that can reach each block
    int2 *fwd, *bwd;          // [lam * nby * nbx], [lam * (nby + 1) / 2 * nbx] listed blocks and pairs of blocks
                              // (candidate, by << 16 | bx): many groups from the front, the others from the back
    float *wp;                // [lam * nbx * nby * kBlkPx] 2 (S - M) (1 - S) / sigma of the listed blocks' pixels
    unsigned *ctl;            // [kCtl] list lengths, tickets, forward exits
    unsigned *rdone;          // [lam] finished blocks of k_soft_reduce
    longlong2 *gv;            // [lam * nI * V]: dL/du, dL/dv in fixed point (units of 2^-36)
    unsigned long long *G;    // [lam * nI * nF * 12][2] fixed point, units of 2^-24 and of 2^-56
    unsigned long long *lsum; // [lam][2] loss in fixed point, units of 2^-41 and of 2^-73
    float *loss;              // [lam]
    float *grad;              // [lam * d] or NULL
};

enum { kFwdHeavy, kFwdLight, kBwdHeavy, kBwdLight, kTicket, kFwdExit = kTicket + 4, kCtl };

// Edge record of a drawable triangle, positively oriented, in image pixels: the
// corners, the edges' unit directions and lengths, and
// +1 / -1 for the mesh's corner order / the reverse, +2 / -2 when all corners
// are on the lattice of 1/256 px.
struct TriRec {
    float x[3], y[3], tx[3], ty[3], L[3], orient;
};

__device__ __forceinline__ TriRec load_rec(const SoftArgs &a, size_t i)
{
    const size_t n = (size_t)a.lam * a.NTp;
    const float4 r0 = a.rec[i], r1 = a.rec[n + i], r2 = a.rec[2 * n + i], r3 = a.rec[3 * n + i];
    TriRec r;
    r.x[0] = r0.x; r.y[0] = r0.y; r.x[1] = r0.z; r.y[1] = r0.w;
    r.x[2] = r1.x; r.y[2] = r1.y; r.tx[0] = r1.z; r.ty[0] = r1.w;
    r.tx[1] = r2.x; r.ty[1] = r2.y; r.tx[2] = r2.z; r.ty[2] = r2.w;
    r.L[0] = r3.x; r.L[1] = r3.y; r.L[2] = r3.z;
    r.orient = r3.w;
    return r;
}

// Kinematics of one instrument of one candidate on warp 0; meanwhile the other
// warps clear the accumulators and count the mask (the loss starts at the
// number of mask pixels: outside every triangle's reach S = 0 and the squared
// error of a pixel is M).
__global__ void __launch_bounds__(kSoftThreads) k_soft_fk(SoftArgs a)
{
    const int c = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    __shared__ int s_m;
    if (tid == 0) s_m = 0;
    __syncthreads();
    const size_t cb = (size_t)c * a.nI + b;
    if (tid < 32) {
        const int dir = lane - 1;
        float st[9];
        for (int k = 0; k < 9; ++k) st[k] = a.params[(size_t)c * a.d + 9 * b + k];
        float T[kMaxFrames][12], dT[kMaxFrames][12];
        if (lane < 10) {
            fk_tangent(a.ch, st, dir, T, dT);
            if (lane == 0)
                for (int f = 0; f < a.nF; ++f)
                    for (int e = 0; e < 12; ++e) a.Tf[(cb * a.nF + f) * 12 + e] = T[f][e];
            else
                for (int f = 0; f < a.nF; ++f)
                    for (int e = 0; e < 12; ++e) a.dT[((cb * a.nF + f) * 9 + dir) * 12 + e] = dT[f][e];
        }
    } else {
        const int t = tid - 32, nt = kSoftThreads - 32;
        if (c == 0 && b == 0 && t < kCtl) a.ctl[t] = 0u;
        if (b == 0) {
            int *cnt = a.count + (size_t)c * a.nby * a.nbx;
            for (int i = t; i < a.nby * a.nbx; i += nt) cnt[i] = 0;
            for (int i = t; i < a.nsup; i += nt)
                a.swin[(size_t)c * a.nsup + i] = make_int4(INT_MAX, INT_MAX, INT_MIN, INT_MIN);
            int m = 0;
            for (int i = t; i < a.H * a.Wq; i += nt) m += __popc(a.mask[i]);
            m = __reduce_add_sync(0xffffffffu, m);
            if (lane == 0) atomicAdd(&s_m, m);
            if (t == 0) a.rdone[c] = 0u;
        }
        if (a.grad) {
            for (int v = t; v < a.V; v += nt) a.gv[cb * a.V + v] = make_longlong2(0, 0);
            for (int e = t; e < a.nF * 24; e += nt) a.G[cb * a.nF * 24 + e] = 0ull;
        }
    }
    __syncthreads();
    if (b == 0 && tid < 2) a.lsum[2 * c + tid] = tid ? 0ull : (unsigned long long)s_m << kLossBits;
}

// Projection of a mesh vertex: (u - cx, v - cy, Z, flag).  Explicit roundings:
// the kernels that call it get the same bits.
__device__ __forceinline__ float4 soft_project(const SoftArgs &a, const float *M, float4 p)
{
    const float X = __fmaf_rn(M[0], p.x, __fmaf_rn(M[1], p.y, __fmaf_rn(M[2], p.z, M[3])));
    const float Y = __fmaf_rn(M[4], p.x, __fmaf_rn(M[5], p.y, __fmaf_rn(M[6], p.z, M[7])));
    const float Z = __fmaf_rn(M[8], p.x, __fmaf_rn(M[9], p.y, __fmaf_rn(M[10], p.z, M[11])));
    float4 o = make_float4(0.0f, 0.0f, Z, 1.0f);
    if (Z >= a.z_near) {
        o.x = __fdiv_rn(__fmul_rn(a.fx, X), Z);
        o.y = __fdiv_rn(__fmul_rn(a.fy, Y), Z);
        if (fabsf(o.x) <= a.guard && fabsf(o.y) <= a.guard) o.w = 0.0f;
    }
    return o;
}

// x to the lattice of 1/256 px (|x| < 2^14; coarser beyond).
__device__ __forceinline__ float rint256(float x) { return __fadd_rn(__fadd_rn(x, 49152.0f), -49152.0f); }

// A warp per group of 32 triangles.  Every lane projects its triangle's three
// corners itself: cheaper than a pass of its own over the vertices and a gather.
__global__ void __launch_bounds__(kSoftThreads) k_soft_tris(SoftArgs a)
{
    const int c = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    extern __shared__ float sT[];  // [nI * nF * 12]
    for (int e = tid; e < a.nI * a.nF * 12; e += kSoftThreads) sT[e] = a.Tf[(size_t)c * a.nI * a.nF * 12 + e];
    __syncthreads();
    const int g = blockIdx.x * (kSoftThreads / 32) + (tid >> 5);
    if (g >= a.ngroups) return;
    const int t = g * 32 + lane;
    const size_t ti = (size_t)c * a.NTp + t;
    float lox = INFINITY, loy = INFINITY, hix = -INFINITY, hiy = -INFINITY;
    float4 bx4 = make_float4(INFINITY, INFINITY, 0.0f, 0.0f);  // no block is near
    if (t < a.nI * a.T) {
        const int b = t >= a.T;
        const int4 tri = a.tris[t - b * a.T];
        const float4 w0 = a.verts[tri.x], w1 = a.verts[tri.y], w2 = a.verts[tri.z];
        const float *M = sT + b * a.nF * 12;
        const float4 p0 = soft_project(a, M + 12 * (int)w0.w, w0), p1 = soft_project(a, M + 12 * (int)w1.w, w1),
                     p2 = soft_project(a, M + 12 * (int)w2.w, w2);
        const float A = (p1.x - p0.x) * (p2.y - p0.y) - (p1.y - p0.y) * (p2.x - p0.x);
        if (p0.w == 0.0f && p1.w == 0.0f && p2.w == 0.0f && A != 0.0f) {
            float x[3] = {p0.x, A > 0.0f ? p1.x : p2.x, A > 0.0f ? p2.x : p1.x};
            float y[3] = {p0.y, A > 0.0f ? p1.y : p2.y, A > 0.0f ? p2.y : p1.y};
            float tx[3], ty[3], L[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int k1 = k == 2 ? 0 : k + 1;
                const float dx = x[k1] - x[k], dy = y[k1] - y[k];
                L[k] = __fsqrt_rn(fmaf(dx, dx, dy * dy));
                const float il = L[k] > 0.0f ? __frcp_rn(L[k]) : 0.0f;
                tx[k] = dx * il;
                ty[k] = dy * il;
            }
            const size_t n = (size_t)a.lam * a.NTp;
#pragma unroll
            for (int k = 0; k < 3; ++k) {  // the edges come from the offsets, unrounded by the shift
                x[k] += a.cx;
                y[k] += a.cy;
            }
            a.rec[ti] = make_float4(x[0], y[0], x[1], y[1]);
            a.rec[n + ti] = make_float4(x[2], y[2], tx[0], ty[0]);
            a.rec[2 * n + ti] = make_float4(tx[1], ty[1], tx[2], ty[2]);
            bool lattice = true;
#pragma unroll
            for (int k = 0; k < 3; ++k) lattice &= rint256(x[k]) == x[k] && rint256(y[k]) == y[k];
            a.rec[3 * n + ti] = make_float4(L[0], L[1], L[2], (A > 0.0f ? 1.0f : -1.0f) * (lattice ? 2.0f : 1.0f));
            lox = fminf(x[0], fminf(x[1], x[2]));
            hix = fmaxf(x[0], fmaxf(x[1], x[2]));
            loy = fminf(y[0], fminf(y[1], y[2]));
            hiy = fmaxf(y[0], fmaxf(y[1], y[2]));
            bx4 = make_float4(0.5f * (lox + hix), 0.5f * (loy + hiy), 0.5f * (hix - lox), 0.5f * (hiy - loy));
        }
    }
    a.box[ti] = bx4;
    for (int o = 16; o; o >>= 1) {
        lox = fminf(lox, __shfl_xor_sync(0xffffffffu, lox, o));
        loy = fminf(loy, __shfl_xor_sync(0xffffffffu, loy, o));
        hix = fmaxf(hix, __shfl_xor_sync(0xffffffffu, hix, o));
        hiy = fmaxf(hiy, __shfl_xor_sync(0xffffffffu, hiy, o));
    }
    short4 win = make_short4(1, 1, 0, 0);
    if (lox <= hix) {
        const float m = kSoftCutoff * a.sigma;
        const int j0 = max(0, (int)floorf(lox - m)), j1 = min(a.W - 1, (int)ceilf(hix + m));
        const int i0 = max(0, (int)floorf(loy - m)), i1 = min(a.H - 1, (int)ceilf(hiy + m));
        if (j0 <= j1 && i0 <= i1)
            win = make_short4((short)(j0 / kBlkW), (short)(i0 / kBlkH), (short)(j1 / kBlkW), (short)(i1 / kBlkH));
    }
    if (lane == 0) a.gwin[(size_t)c * a.ngroups + g] = win;
    if (win.x > win.z) return;
    if (lane < 4) {
        int *sw = reinterpret_cast<int *>(a.swin + (size_t)c * a.nsup + (g >> 5)) + lane;
        if (lane < 2) atomicMin(sw, lane ? win.y : win.x);
        else atomicMax(sw, lane == 3 ? win.w : win.z);
    }
    const int bw = win.z - win.x + 1, nb = bw * (win.w - win.y + 1);
    int *cnt = a.count + ((size_t)c * a.nby + win.y) * a.nbx + win.x;
    for (int e = lane; e < nb; e += 32) atomicAdd(cnt + (e / bw) * a.nbx + e % bw, 1);
}

// The work lists: a thread per pair of blocks (a block and the one below).
__device__ __forceinline__ void append(const SoftArgs &a, bool on, bool heavy, int2 v, int base, int2 *list, int cap)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const bool take = on && heavy == (h == 0);
        const unsigned m = __ballot_sync(0xffffffffu, take);
        if (!m) continue;
        const int lane = threadIdx.x & 31;
        unsigned at = 0;
        if (lane == __ffs(m) - 1) at = atomicAdd(&a.ctl[base + h], (unsigned)__popc(m));
        at = __shfl_sync(0xffffffffu, at, __ffs(m) - 1) + __popc(m & ((1u << lane) - 1u));
        if (take) list[h == 0 ? at : cap - 1 - at] = v;
    }
}

__global__ void __launch_bounds__(kSoftThreads) k_soft_list(SoftArgs a)
{
    const int c = blockIdx.y, i = blockIdx.x * kSoftThreads + threadIdx.x, nby2 = (a.nby + 1) / 2;
    const int by = 2 * (i / a.nbx), bx = i % a.nbx;
    const bool in = i < nby2 * a.nbx;
    const int *cnt = a.count + ((size_t)c * a.nby + by) * a.nbx + bx;
    const int n0 = in ? cnt[0] : 0, n1 = in && by + 1 < a.nby ? cnt[a.nbx] : 0;
    const int2 v0 = make_int2(c, by << 16 | bx), v1 = make_int2(c, (by + 1) << 16 | bx);
    const int cap = a.lam * a.nby * a.nbx;
    append(a, n0 > 0, n0 >= a.heavy, v0, kFwdHeavy, a.fwd, cap);
    append(a, n1 > 0, n1 >= a.heavy, v1, kFwdHeavy, a.fwd, cap);
    if (a.grad) append(a, n0 + n1 > 0, max(n0, n1) >= a.heavy, v0, kBwdHeavy, a.bwd, a.lam * nby2 * a.nbx);
}

// The entries of a kernel's list: the heavy ones are taken by the whole block
// (a ticket through shared memory), then the light ones by each warp for
// itself.  The next ticket is drawn while the entry before it is worked on.
struct Work {
    bool heavy = true;
    int c = 0, bx = 0, by = 0;
    int ticket = 0, n_heavy, n_light;  // the ticket: thread 0's, later each warp's lane 0's

    __device__ __forceinline__ Work(const SoftArgs &a, int base) : n_heavy((int)a.ctl[base]), n_light((int)a.ctl[base + 1])
    {
        if (threadIdx.x == 0) ticket = (int)atomicAdd(&a.ctl[kTicket + base], 1u);
    }

    __device__ __forceinline__ void take(int2 v) { c = v.x, bx = v.y & 0xffff, by = v.y >> 16; }

    __device__ __forceinline__ bool next(const SoftArgs &a, int base, const int2 *list, int cap, int *s_it)
    {
        const int lane = threadIdx.x & 31;
        if (heavy) {
            __syncthreads();  // the previous entry's shared memory is free
            if (threadIdx.x == 0) {
                *s_it = ticket;
                if (ticket < n_heavy) ticket = (int)atomicAdd(&a.ctl[kTicket + base], 1u);
            }
            __syncthreads();
            const int i = *s_it;
            if (i < n_heavy) {
                take(list[i]);
                return true;
            }
            heavy = false;
            if (lane == 0) ticket = (int)atomicAdd(&a.ctl[kTicket + base + 1], 1u);
        }
        const int i = __shfl_sync(0xffffffffu, ticket, 0);
        if (i >= n_light) return false;
        if (lane == 0) ticket = (int)atomicAdd(&a.ctl[kTicket + base + 1], 1u);
        take(list[cap - 1 - i]);
        return true;
    }
};

__device__ __forceinline__ float min3(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float ex2(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float sqrt_(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsq(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// |x| with the sign of s
__device__ __forceinline__ float with_sign(float x, float s)
{
    return __uint_as_float(__float_as_uint(x) | (__float_as_uint(s) & 0x80000000u));
}

// The triangles that come within the cutoff of `kRows` rows of pixels from block
// (bx, by) down, collected into batches of 32 by one warp.  Runs of 32 groups,
// then groups (of those the ones whose number is `warp` modulo nw), then
// triangles are tested against the block, one per lane; the next group's boxes
// and the next batch's records are on their way while the last are used.
template <int kRows>
struct Collector {
    const int4 *sw;    // the candidate's windows of runs and groups, boxes and records
    const short4 *gw;
    const float4 *box, *rec;
    size_t stride;
    int *qu;           // the warp's queue (64 entries)
    int bx, by, s0 = 0, sb = 0, gb = 0, qn = 0, nsup, ngroups;
    unsigned sup = 0, hits = 0, mine;
    float reach2;
    float4 pre;        // box of the next group's triangle

    __device__ __forceinline__ Collector(const SoftArgs &a, int c, int bx_, int by_, int warp, int nw, int *queue)
        : sw(a.swin + (size_t)c * a.nsup), gw(a.gwin + (size_t)c * a.ngroups), box(a.box + (size_t)c * a.NTp),
          rec(a.rec + (size_t)c * a.NTp), stride((size_t)a.lam * a.NTp), qu(queue), bx(bx_), by(by_), nsup(a.nsup),
          ngroups(a.ngroups), mine(nw == 1 ? 0xffffffffu : 0x11111111u << warp)
    {
        static_assert(kFwdWarps == 4 && kBwdWarps == 4, "`mine` takes every fourth group");
        const float reach = kSoftCutoff * a.sigma + 0.01f;
        reach2 = reach * reach;
    }

    __device__ __forceinline__ bool near(float4 b) const
    {
        const float x = (float)(bx * kBlkW) + 0.5f * (kBlkW - 1), y = (float)(by * kBlkH) + 0.5f * (kRows - 1);
        const float dx = fmaxf(fabsf(b.x - x) - (b.z + 0.5f * (kBlkW - 1)), 0.0f);
        const float dy = fmaxf(fabsf(b.y - y) - (b.w + 0.5f * (kRows - 1)), 0.0f);
        return fmaf(dx, dx, dy * dy) <= reach2;
    }

    __device__ __forceinline__ bool in(int x0, int y0, int x1, int y1) const
    {
        return x0 <= bx && bx <= x1 && y0 <= by + (kRows - 1) / kBlkH && by <= y1;
    }

    // The next batch: the lane's triangle (numbered within the candidate) or
    // -1; false when no triangle is left.
    __device__ __forceinline__ bool next(int lane, int &t)
    {
        while (qn < 32) {
            if (!hits) {
                if (!sup) {
                    if (s0 >= nsup) break;
                    sb = s0;
                    bool h = false;
                    if (sb + lane < nsup) {
                        const int4 w = sw[sb + lane];
                        h = in(w.x, w.y, w.z, w.w);
                    }
                    sup = __ballot_sync(0xffffffffu, h);
                    s0 += 32;
                    continue;
                }
                gb = (sb + __ffs(sup) - 1) * 32;
                sup &= sup - 1;
                bool h = false;
                if (gb + lane < ngroups) {
                    const short4 w = gw[gb + lane];
                    h = in(w.x, w.y, w.z, w.w);
                }
                hits = __ballot_sync(0xffffffffu, h) & mine;
                if (hits) pre = box[(gb + __ffs(hits) - 1) * 32 + lane];
                continue;
            }
            const int tt = (gb + __ffs(hits) - 1) * 32 + lane;
            const float4 b = pre;
            hits &= hits - 1;
            if (hits) pre = box[(gb + __ffs(hits) - 1) * 32 + lane];
            const bool h = near(b);
            const unsigned m = __ballot_sync(0xffffffffu, h);
            if (h) qu[qn + __popc(m & ((1u << lane) - 1u))] = tt;
            qn += __popc(m);
        }
        if (qn == 0) return false;
        __syncwarp();
        const int n = min(qn, 32);  // the last (up to) 32 of the queue
        qn -= n;
        t = lane < n ? qu[qn + lane] : -1;
        __syncwarp();
        if (t >= 0)
#pragma unroll
            for (int q = 0; q < 4; ++q) asm volatile("prefetch.global.L1 [%0];" ::"l"(rec + q * stride + t));
        return true;
    }
};

// The edges of a triangle seen from a block, in units of the cutoff (14 sigma):
// the coordinates of the row's first pixel along each edge from its middle (a)
// and across it (b, positive inside), the edge's direction and half its length.
// In these units a point's distance beyond an edge's end, |a| - h clamped to
// [0, 1], is one saturating addition: what is clamped at 1 is out of reach.
// (FP32 additions and FMAs issue every cycle, minima, selections and logic
// every second one, packed FP32 pairs take two cycles: a version on pairs of
// pixels was no faster.)
struct BlockEdges {
    float a[3], b[3], tx[3], ty[3], h[3];

    __device__ __forceinline__ void down()  // to the next row of pixels
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a[k] += ty[k];
            b[k] += tx[k];
        }
    }
};

__device__ __forceinline__ BlockEdges block_edges(const TriRec &r, bool drawn, int bx, int by, float unit)
{
    const float X = (float)(bx * kBlkW), Y = (float)(by * kBlkH);
    BlockEdges e;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float rx = X - r.x[q], ry = Y - r.y[q];
        e.tx[q] = drawn ? r.tx[q] * unit : 0.0f;
        e.ty[q] = drawn ? r.ty[q] * unit : 0.0f;
        e.h[q] = 0.5f * r.L[q] * unit;
        e.a[q] = fmaf(rx, e.tx[q], ry * e.ty[q]) - e.h[q];
        e.b[q] = drawn ? fmaf(ry, e.tx[q], -rx * e.ty[q]) : -10.0f;  // no triangle: out of reach
    }
    return e;
}

constexpr float kExpScale = kSoftCutoff * 1.44269504089f;  // exp(d / sigma) = 2^(kExpScale d / cutoff)

// The product over one batch of triangles (one per lane) into the lane's 32
// running products Q (1 + Q = product of 1 + exp(d / sigma)).  Per pixel: the
// point's coordinates (a, b) in the three edge frames, the squared distance
// b^2 + max(|a| - h, 0)^2 to each edge, its minimum, the sign from the smallest
// b (inside: every b >= 0, and there the nearest edge's line is nearest at the
// edge), and one exponential.
__device__ __forceinline__ void fwd_batch(BlockEdges &e, float (&Q)[kBlkPx])
{
#pragma unroll
    for (int py = 0; py < kBlkH; ++py) {
        // stage by stage over a row, so that eight pixels are in flight
        float d[kBlkW], sg[kBlkW];
#pragma unroll
        for (int px = 0; px < kBlkW; ++px) {
            float d2[3], b[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float a = fmaf((float)px, e.tx[k], e.a[k]);
                b[k] = fmaf(-(float)px, e.ty[k], e.b[k]);
                const float o = __saturatef(fabsf(a) - e.h[k]);
                d2[k] = fmaf(o, o, b[k] * b[k]);
            }
            d[px] = min3(d2[0], d2[1], d2[2]);
            sg[px] = min3(b[0], b[1], b[2]);
        }
#pragma unroll
        for (int px = 0; px < kBlkW; ++px) d[px] = with_sign(sqrt_(d[px]), sg[px]);
#pragma unroll
        for (int px = 0; px < kBlkW; ++px) sg[px] = ex2(d[px] * kExpScale);
#pragma unroll
        for (int px = 0; px < kBlkW; ++px) {
            float &q = Q[py * kBlkW + px];
            if (d[px] > -1.0f) q = fmaf(q, sg[px], q + sg[px]);  // q > 0: an infinite term makes q infinite, never NaN
        }
        e.down();
    }
}

// The lanes' products multiplied together: returns pixel `lane`'s.
__device__ __forceinline__ float combine_lanes(const float (&Q)[kBlkPx], int lane)
{
    float v[16];
    {
        const bool up = lane & 16;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float mine = up ? Q[i + 16] : Q[i], give = up ? Q[i] : Q[i + 16];
            const float got = __shfl_xor_sync(0xffffffffu, give, 16);
            v[i] = fmaf(mine, got, mine + got);
        }
    }
#pragma unroll
    for (int s = 8; s; s >>= 1) {
        const bool up = lane & s;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < s) {
                const float mine = up ? v[i + s] : v[i], give = up ? v[i] : v[i + s];
                const float got = __shfl_xor_sync(0xffffffffu, give, s);
                v[i] = fmaf(mine, got, mine + got);
            }
    }
    return v[0];
}

// Persistent blocks over the listed pixel blocks.  A light block of pixels is
// one warp's (no barrier, at most one batch that is not full); a heavy one (a
// shaft seen end-on puts thousands of triangles within its reach) is shared by
// the block's warps, every fourth group to a warp.  Bound by issue (65 % of the
// cycles; half of the instructions evaluate pairs, a third collect them).  The
// loss of 64 candidates at 640x512, 20k triangles, takes 0.61 and 0.67 ms in two
// scenes and 1.57 ms in one seen end-on.  With every block shared by four warps
// this kernel takes 1.3 to 1.8 times as long; with one warp each about as long,
// but then 8 candidates, where the heaviest blocks decide, take half as long again
// for a loss and a gradient.  (A pixel per thread with the triangles in shared
// memory, about 180 instructions per pair, was 8 to 20 times slower.)
// Every kCheck batches a warp looks whether the pixels are saturated (see
// kSaturated) by its own products and the last ones the other warps left in
// shared memory: those only grow, so a decision made on them holds, and the
// results do not depend on when it is made.
__global__ void __launch_bounds__(32 * kFwdWarps, 5) k_soft_fwd(SoftArgs a)
{
    constexpr int kCheck = 6;
    __shared__ int queue[kFwdWarps][64];
    __shared__ float part[kFwdWarps][kBlkPx];
    __shared__ int s_it;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float unit = 1.0f / (kSoftCutoff * a.sigma), inv_s = 1.0f / a.sigma;
    Work w(a, kFwdHeavy);
    while (w.next(a, kFwdHeavy, a.fwd, a.lam * a.nby * a.nbx, &s_it)) {
        const int c = w.c;
        const size_t tb = (size_t)c * a.NTp;
        const int j = w.bx * kBlkW + (lane & (kBlkW - 1)), i = w.by * kBlkH + lane / kBlkW;
        const bool on = j < a.W && i < a.H;
        if (w.heavy) {
            part[warp][lane] = kEmpty;
            __syncthreads();
        }
        float Q[kBlkPx];
#pragma unroll
        for (int p = 0; p < kBlkPx; ++p) Q[p] = kEmpty;
        Collector<kBlkH> col(a, c, w.bx, w.by, warp, w.heavy ? kFwdWarps : 1, queue[warp]);
        int t, batches = 0;
        bool more = col.next(lane, t);
        while (more) {
            BlockEdges e = block_edges(load_rec(a, tb + max(t, 0)), t >= 0, w.bx, w.by, unit);
            more = col.next(lane, t);
            fwd_batch(e, Q);
            if (++batches % kCheck == 0) {
                float q = combine_lanes(Q, lane);
                if (w.heavy) {
                    part[warp][lane] = q;
                    volatile float(*pv)[kBlkPx] = part;
#pragma unroll
                    for (int o = 1; o < kFwdWarps; ++o) {
                        const float r = pv[(warp + o) % kFwdWarps][lane];
                        q = fmaf(q, r, q + r);
                    }
                }
                if (__all_sync(0xffffffffu, !on || q >= kSaturated)) break;
            }
        }
        float q = combine_lanes(Q, lane);
        if (w.heavy) {
            part[warp][lane] = q;
            __syncthreads();
            if (warp) continue;
            for (int o = 1; o < kFwdWarps; ++o) {
                const float r = part[o][lane];
                q = fmaf(q, r, q + r);
            }
        }
        float l = 0.0f, wpx = 0.0f;
        const bool mv = on && ((a.mask[(size_t)i * a.Wq + (j >> 5)] >> (j & 31)) & 1u);
        if (on) {
            const bool sat = q >= kOne;
            const float om = sat ? 0.0f : __frcp_rn(1.0f + q);  // 1 - S
            const float S = sat ? 1.0f : q * om;
            const float e = mv ? -om : S;
            l = e * e;
            wpx = 2.0f * e * om * inv_s;
        }
        if (a.grad) a.wp[(((size_t)c * a.nby + w.by) * a.nbx + w.bx) * kBlkPx + lane] = wpx;
        const int m = __popc(__ballot_sync(0xffffffffu, mv));
        for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) {  // squared error minus the mask pixels counted in advance: exact sums, in any order
            const float q = l * kLossScale, h = rintf(q);
            const long long rest = to_fixed(q - h, kRestScale);
            atomicAdd(a.lsum + 2 * c, (unsigned long long)__float2ll_rn(h) - ((unsigned long long)m << kLossBits));
            if (rest) atomicAdd(a.lsum + 2 * c + 1, (unsigned long long)rest);
        }
    }
    // the last block to run out of work writes the losses
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_it = atomicAdd(&a.ctl[kFwdExit], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_it) {
        __threadfence();
        for (int c = tid; c < a.lam; c += blockDim.x)
            a.loss[c] = (float)(((double)(long long)__ldcg(a.lsum + 2 * c) +
                                 (double)(long long)__ldcg(a.lsum + 2 * c + 1) * (1.0 / kRestScale)) * (1.0 / kLossScale));
    }
}

// dL/d(u, v) of the triangles over two blocks of pixels, one triangle per lane.
// With c the closest boundary point, at parameter t of edge k, the signed
// distance d changes with c by -(p - c) / d, and c follows the edge's ends by
// 1 - t and t.  The sums are kept in the edges' frames: the parts along the
// edge (only beyond an end: U, and V signed by the end) and across it (W, and Wt
// weighted by the position of c on the edge, from its middle).
// On the boundary p - c and d vanish together, but d is smooth there and the
// derivative is their limit, one unit along the edge's normal: within kOnEdge of
// an edge (in units of the cutoff: 3e-5 sigma, and more than FP32 leaves of the
// distance of a centre that lies on the edge of a triangle some hundred pixels
// across) the part across is the weight itself.  Where the derivative jumps (a
// centre on a corner, or as far from two edges) the first of the nearest edges
// takes the pixel, as in a comparison without rounding: squared distances count
// as equal within kOnEdge^2, and for a triangle with all corners on the lattice of
// 1/256 px, whose bisectors run through pixel centres, within the rounding's part,
// kTie h for edges of half length h.  Of other triangles the nearest edge counts as
// FP32 has it: a margin assigned more pixels to the wrong edge than it put right
// (gradients of 20k triangles 1.0e-6 -> 5.0e-6 from 64 bits at worst).
// The blocks are the forward's, two at a time (half the atomic additions for a
// few more idle lanes); light and heavy ones as there.  Bound by issue (67 % of
// the cycles); a loss and its gradient in the forward's three scenes: 1.75, 2.05
// and 4.43 ms.  With the groups walking the whole of their windows, one set of
// additions per triangle, 18-21 % of the lanes had a pair within reach (here
// 60 %) and this kernel took 2.2 times as long.
struct EdgeSums {
    float U[3], V[3], W[3], Wt[3];
};
constexpr float kOnEdge = 1.0f / 524288.0f, kTie = 1.0f / 65536.0f;

__device__ __forceinline__ void bwd_pixel(const BlockEdges &e, int px, float w, float tie, EdgeSums &s)
{
    float d2[3], b[3], over[3], o[3], f[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float a = fmaf((float)px, e.tx[k], e.a[k]);
        b[k] = fmaf(-(float)px, e.ty[k], e.b[k]);
        over[k] = __saturatef(fabsf(a) - e.h[k]);
        d2[k] = fmaf(over[k], over[k], fmaf(b[k], b[k], 1e-30f));  // never zero
        o[k] = with_sign(over[k], a);
        f[k] = a - o[k];
    }
    const float m = min3(d2[0], d2[1], d2[2]);
    const float ir = with_sign(rsq(m), min3(b[0], b[1], b[2]));
    const float d = m * ir;
    const float sg = rcp_(1.0f + ex2(d * -kExpScale));
    // outside: d = -|p - c|, the sum grows along p - c; inside the other way
    const bool on = m <= kOnEdge * kOnEdge;
    const float q = w * sg;
    const float v = on ? 0.0f : q * -ir, across = on ? -q : 0.0f;
    const float nearest = fmaf(m, tie, kOnEdge * kOnEdge);
    // the nearest edge (the first of equal ones) takes it, none beyond the cutoff
    asm("{\n\t"
        ".reg .pred in, p0, r, p1, p2;\n\t"
        ".reg .f32 x;\n\t"
        "setp.gt.f32 in, %12, 0fBF800000;\n\t"
        "setp.le.and.f32 p0|r, %13, %16, in;\n\t"
        "setp.le.and.f32 p1|p2, %14, %16, r;\n\t"
        "@p0 fma.rn.f32 %0, %17, %18, %0;\n\t"
        "@p0 fma.rn.f32 %3, %17, %19, %3;\n\t"
        "@p0 fma.rn.f32 x, %17, %20, %15;\n\t"
        "@p0 add.f32 %6, %6, x;\n\t"
        "@p0 fma.rn.f32 %9, x, %21, %9;\n\t"
        "@p1 fma.rn.f32 %1, %17, %22, %1;\n\t"
        "@p1 fma.rn.f32 %4, %17, %23, %4;\n\t"
        "@p1 fma.rn.f32 x, %17, %24, %15;\n\t"
        "@p1 add.f32 %7, %7, x;\n\t"
        "@p1 fma.rn.f32 %10, x, %25, %10;\n\t"
        "@p2 fma.rn.f32 %2, %17, %26, %2;\n\t"
        "@p2 fma.rn.f32 %5, %17, %27, %5;\n\t"
        "@p2 fma.rn.f32 x, %17, %28, %15;\n\t"
        "@p2 add.f32 %8, %8, x;\n\t"
        "@p2 fma.rn.f32 %11, x, %29, %11;\n\t"
        "}"
        : "+f"(s.U[0]), "+f"(s.U[1]), "+f"(s.U[2]), "+f"(s.V[0]), "+f"(s.V[1]), "+f"(s.V[2]), "+f"(s.W[0]),
          "+f"(s.W[1]), "+f"(s.W[2]), "+f"(s.Wt[0]), "+f"(s.Wt[1]), "+f"(s.Wt[2])
        : "f"(d), "f"(d2[0]), "f"(d2[1]), "f"(across), "f"(nearest), "f"(v), "f"(o[0]), "f"(over[0]), "f"(b[0]),
          "f"(f[0]), "f"(o[1]), "f"(over[1]), "f"(b[1]), "f"(f[1]), "f"(o[2]), "f"(over[2]), "f"(b[2]), "f"(f[2]));
}

constexpr int kBwdRows = 2 * kBlkH;  // the backward takes a block and the one below

__global__ void __launch_bounds__(32 * kBwdWarps, 5) k_soft_bwd(SoftArgs a)
{
    __shared__ int queue[kBwdWarps][64];
    __shared__ float s_w[kBwdWarps][kBwdRows * kBlkW];
    __shared__ int s_it;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float unit = 1.0f / (kSoftCutoff * a.sigma);
    Work w(a, kBwdHeavy);
    while (w.next(a, kBwdHeavy, a.bwd, a.lam * ((a.nby + 1) / 2) * a.nbx, &s_it)) {
        const int c = w.c;
        float *sw = s_w[warp];  // the pixels' factors, a copy for every warp
        unsigned nzh[2];
        const size_t blk = ((size_t)c * a.nby + w.by) * a.nbx + w.bx;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const size_t q = blk + (size_t)h * a.nbx;
            const float v = w.by + h < a.nby && a.count[q] > 0 ? a.wp[q * kBlkPx + lane] : 0.0f;
            sw[h * kBlkPx + lane] = v;
            nzh[h] = __ballot_sync(0xffffffffu, v != 0.0f);
        }
        const unsigned long long nz = (unsigned long long)nzh[1] << 32 | nzh[0];
        if (!nz) continue;
        __syncwarp();
        const size_t tb = (size_t)c * a.NTp;
        Collector<kBwdRows> col(a, c, w.bx, w.by, warp, w.heavy ? kBwdWarps : 1, queue[warp]);
        int tn;
        bool more = col.next(lane, tn);
        while (more) {
            const int t = tn;
            const TriRec r = load_rec(a, tb + max(t, 0));
            more = col.next(lane, tn);
            BlockEdges e = block_edges(r, t >= 0, w.bx, w.by, unit);
            const float tie = fabsf(r.orient) > 1.0f ? fmaf(kTie, fmaxf(e.h[0], fmaxf(e.h[1], e.h[2])), 1.0f) : 1.0f;
            EdgeSums s{};
            for (int py = 0; py < kBwdRows; ++py) {
                const unsigned row = (unsigned)(nz >> (kBlkW * py)) & ((1u << kBlkW) - 1u);
                if (row) {
#pragma unroll
                    for (int px = 0; px < kBlkW; ++px)
                        if (row >> px & 1u) bwd_pixel(e, px, sw[kBlkW * py + px], tie, s);
                }
                e.down();
            }
            if (t < 0) continue;
            float gx[3] = {0.0f, 0.0f, 0.0f}, gy[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int k1 = k == 2 ? 0 : k + 1;
                const float h = 0.5f * r.L[k] * unit, i2h = h > 0.0f ? 0.5f / h : 0.0f;
                // the ends' shares: t = (f + h) / 2h, and what is left; beyond an end t is 0 or 1
                const float u1 = 0.5f * (s.U[k] + s.V[k]), u0 = s.U[k] - u1;
                const float w1 = fmaf(h, s.W[k], s.Wt[k]) * i2h, w0 = s.W[k] - w1;
                gx[k] += r.tx[k] * u0 - r.ty[k] * w0;
                gy[k] += r.ty[k] * u0 + r.tx[k] * w0;
                gx[k1] += r.tx[k] * u1 - r.ty[k] * w1;
                gy[k1] += r.ty[k] * u1 + r.tx[k] * w1;
            }
            const int b = t >= a.T;
            const int4 tri = a.tris[t - b * a.T];
            const int id[3] = {tri.x, r.orient > 0.0f ? tri.y : tri.z, r.orient > 0.0f ? tri.z : tri.y};
#pragma unroll
            for (int k = 0; k < 3; ++k) {  // fixed point: the sums do not depend on the order of the additions
                unsigned long long *gp =
                    reinterpret_cast<unsigned long long *>(a.gv + ((size_t)c * a.nI + b) * a.V + id[k]);
                const long long vx = to_fixed(gx[k], kGvScale), vy = to_fixed(gy[k], kGvScale);
                if (vx) atomicAdd(gp, (unsigned long long)vx);
                if (vy) atomicAdd(gp + 1, (unsigned long long)vy);
            }
        }
    }
}

// Per (candidate, instrument): dL/dX of every vertex, G_f = sum over the
// frame's vertices of dL/dX [v; 1]^T; the candidate's last block contracts
// dL/dtheta_k = sum_f <G_f, dT_f/dtheta_k>.  The sums are fixed-point integers,
// so a call's results do not vary from run to run.  A warp takes 64
// consecutive vertices (mostly of one frame: a link's vertices are contiguous),
// two per lane.
constexpr int kRedVerts = 2;

__global__ void __launch_bounds__(kSoftThreads) k_soft_reduce(SoftArgs a)
{
    const int c = blockIdx.y / a.nI, b = blockIdx.y % a.nI, tid = threadIdx.x, lane = tid & 31;
    __shared__ int s_last;
    const size_t cb = (size_t)c * a.nI + b;
    const float *Tf = a.Tf + cb * a.nF * 12;
    unsigned long long *G = a.G + cb * a.nF * 24;
    long long acc[24];
#pragma unroll
    for (int k = 0; k < 24; ++k) acc[k] = 0;
    int fcur = -1;
    auto flush = [&]() {
        if (fcur < 0) return;
#pragma unroll
        for (int k = 0; k < 24; ++k) {
            if (acc[k]) atomicAdd(G + fcur * 24 + k, (unsigned long long)acc[k]);
            acc[k] = 0;
        }
    };
    auto add = [&](int k, float x) {  // the whole units and the rest, both exact
        const float q = x * kGScale, h = rintf(q);
        acc[2 * k] += __float2ll_rn(h);
        acc[2 * k + 1] += __float2ll_rn((q - h) * kRestScale);
    };
    const int v0 = ((int)blockIdx.x * kSoftThreads + (tid & ~31)) * kRedVerts + lane;
#pragma unroll
    for (int q = 0; q < kRedVerts; ++q) {
        const int v = v0 + 32 * q;
        if (v >= a.V) break;
        const longlong2 gq = a.gv[cb * a.V + v];
        if (gq.x == 0 && gq.y == 0) continue;
        const float4 p = a.verts[v];
        const int f = (int)p.w;
        const float4 s = soft_project(a, Tf + 12 * f, p);
        const float gx = __ll2float_rn(gq.x) * (1.0f / kGvScale), gy = __ll2float_rn(gq.y) * (1.0f / kGvScale);
        const float iz = 1.0f / s.z;
        const float gX = gx * a.fx * iz, gY = gy * a.fy * iz, gZ = -(gx * s.x + gy * s.y) * iz;
        if (f != fcur) {
            flush();
            fcur = f;
        }
        const float vh[4] = {p.x, p.y, p.z, 1.0f};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            add(k, gX * vh[k]);
            add(4 + k, gY * vh[k]);
            add(8 + k, gZ * vh[k]);
        }
    }
    // one frame in the whole warp: one addition per entry instead of 32
    const int fw = __reduce_max_sync(0xffffffffu, fcur);
    if (__all_sync(0xffffffffu, fcur == fw || fcur < 0)) {
        if (fw >= 0) {
#pragma unroll
            for (int k = 0; k < 24; ++k)
                for (int o = 16; o; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
            if (lane == 0) {
                fcur = fw;
                flush();
            }
        }
    } else {
        flush();
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(a.rdone + c, 1u) == gridDim.x * a.nI - 1;
    }
    __syncthreads();
    if (!s_last || tid >= 9 * a.nI) return;
    __threadfence();
    const int bb = tid / 9, k = tid - 9 * bb;
    const size_t cbb = (size_t)c * a.nI + bb;
    float sum = 0.0f;
    for (int f = 0; f < a.nF; ++f)
#pragma unroll
        for (int e = 0; e < 12; ++e) {
            const unsigned long long *g = a.G + ((cbb * a.nF + f) * 12 + e) * 2;
            const float gv = fmaf(__ll2float_rn((long long)__ldcg(g + 1)), 1.0f / kRestScale,
                                  __ll2float_rn((long long)__ldcg(g)));
            sum = fmaf(gv * (1.0f / kGScale), a.dT[((cbb * a.nF + f) * 9 + k) * 12 + e], sum);
        }
    a.grad[(size_t)c * a.d + 9 * bb + k] = sum;
}

// Adam on the refined candidates, in the optimiser's normalised units
// (x = params / scales): m, v, bias correction (Kingma & Ba, 2015).
__global__ void k_adam(float *P, const float *g, float *m, float *v, const CmaConst *k, int n, int d, float lr,
                       float b1, float b2, float eps, int step)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * d) return;
    const float sc = (float)k->scales[i % d];
    const float gn = g[i] * sc;
    const float mi = b1 * m[i] + (1.0f - b1) * gn;
    const float vi = b2 * v[i] + (1.0f - b2) * gn * gn;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / (1.0f - powf(b1, (float)step)), vh = vi / (1.0f - powf(b2, (float)step));
    P[i] -= lr * sc * mh / (sqrtf(vh) + eps);
}

// The k best candidates of the last generation (by loss, then index) into P;
// Adam moments cleared.
__global__ void k_refine_init(const float *params, const float *loss, int lam, int d, int kk, float *P, float *m,
                              float *v, int *order)
{
    __shared__ int sel[32];
    if (threadIdx.x == 0) {
        for (int r = 0; r < kk; ++r) {
            int best = -1;
            for (int c = 0; c < lam; ++c) {
                bool taken = false;
                for (int q = 0; q < r; ++q) taken |= sel[q] == c;
                if (taken) continue;
                if (best < 0 || loss[c] < loss[best]) best = c;  // ties keep the lower index
            }
            sel[r] = best;
            order[r] = best;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kk * d; e += blockDim.x) {
        P[e] = params[(size_t)sel[e / d] * d + e % d];
        m[e] = 0.0f;
        v[e] = 0.0f;
    }
}

// The refined candidate with the lowest fitness loss (ties: lower index)
// replaces the frame's estimate when it beats the frame's best.
__global__ void k_refine_pick(const float *P, const float *lhard, int kk, int d, CmaState *st, float *pose_out,
                              int *picked)
{
    __shared__ int best;
    if (threadIdx.x == 0) {
        int b = 0;
        for (int r = 1; r < kk; ++r)
            if (lhard[r] < lhard[b]) b = r;
        best = (lhard[b] < st->best_loss) ? b : -1;
        *picked = best;
        if (best >= 0) st->best_loss = lhard[b];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        if (best >= 0) {
            const float x = P[(size_t)best * d + i];
            st->best_x[i] = x;
            st->est[i] = (double)x;
        }
        if (pose_out) pose_out[i] = (float)st->est[i];
    }
}

}  // namespace trk

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
using namespace trk;

namespace {

// Scratch of one tracker: one allocation, which every call lays out for itself.
// It is sized for a gradient whichever kind of call comes first: a gradient on as
// many candidates then finds its memory (it may be under capture, and a captured
// loss may still use what growing would free).
struct SoftScratch {
    size_t bytes = 0;
    int fwd_grid = 0, bwd_grid = 0;
    void *mem = nullptr;
};

// A call on more candidates than the scratch holds takes them in slices; it grows
// to two gigabytes, or one candidate's need (the records and the per-pixel
// factors of a 640x512, 20k-triangle candidate are about 3.5 MB).
constexpr size_t kSoftBudget = (size_t)2 << 30;

struct RefineBuf {
    int cap = 0;
    float *P = nullptr, *g = nullptr, *m = nullptr, *v = nullptr, *ls = nullptr, *lh = nullptr;
    int *order = nullptr, *picked = nullptr;
};

trk_status soft_fail(trk_status st, const char *why)
{
    set_last_error(why);
    return st;
}

// Lays the arrays out from `base` (NULL: only counts) and returns the bytes.
size_t soft_layout(SoftArgs &a, int lam, bool grad, char *base)
{
    size_t off = 0;
    auto take = [&](auto *&p, size_t n) {
        p = base ? reinterpret_cast<std::remove_reference_t<decltype(p)>>(base + off) : nullptr;
        off += (n * sizeof(*p) + 255) & ~(size_t)255;
    };
    const size_t L = (size_t)lam, nb = (size_t)a.nbx * a.nby, nt = L * a.NTp, fr = L * a.nI * a.nF;
    take(a.rec, 4 * nt);
    take(a.box, nt);
    take(a.gwin, L * a.ngroups);
    take(a.swin, L * a.nsup);
    take(a.count, L * nb);
    take(a.fwd, L * nb);
    take(a.ctl, kCtl);
    take(a.rdone, L);
    take(a.lsum, 2 * L);
    take(a.Tf, fr * 12);
    take(a.dT, fr * 9 * 12);
    if (grad) {
        take(a.bwd, L * ((a.nby + 1) / 2) * a.nbx);
        take(a.wp, L * nb * kBlkPx);
        take(a.gv, L * a.nI * a.V);
        take(a.G, fr * 24);
    }
    return off;
}

void soft_shape(SoftArgs &a, const trk_tracker *t)
{
    a.ch = t->ch;
    a.nF = t->ch.n_frames;
    a.nI = t->ch.n_inst;
    a.V = t->V;
    a.T = t->T;
    a.d = t->d;
    a.W = t->cam.W;
    a.H = t->cam.H;
    a.Wq = t->cam.Wq;
    a.nbx = (a.W + kBlkW - 1) / kBlkW;
    a.nby = (a.H + kBlkH - 1) / kBlkH;
    a.heavy = a.nbx * a.nby <= kSmallBlocks ? kHeavySmall : kHeavy;
    a.ngroups = (int)(((long long)a.nI * a.T + 31) / 32);
    a.NTp = 32 * a.ngroups;
    a.nsup = (a.ngroups + 31) / 32;
}

// As many candidates (at least one) as `bytes` hold for this kind of call.
int soft_fit(SoftArgs &a, int lam, bool grad, size_t bytes)
{
    return (int)std::max<size_t>(1, std::min<size_t>((size_t)lam, bytes / soft_layout(a, 1, grad, nullptr)));
}

trk_status soft_scratch(trk_tracker *t, size_t bytes, SoftScratch **out)
{
    SoftScratch *s = static_cast<SoftScratch *>(t->soft);
    if (s && s->bytes >= bytes) {
        *out = s;
        return TRK_OK;
    }
    soft_free(t);
    s = new SoftScratch();
    t->soft = s;
    cudaError_t e;
    int fwd = 0, bwd = 0, sms = 0;
    if ((e = cudaMalloc(&s->mem, bytes)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, t->device)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fwd, k_soft_fwd, 32 * kFwdWarps, 0)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bwd, k_soft_bwd, 32 * kBwdWarps, 0)) != cudaSuccess) {
        soft_free(t);
        return soft_fail(e == cudaErrorMemoryAllocation ? TRK_ENOMEM : TRK_ECUDA, cudaGetErrorString(e));
    }
    s->bytes = bytes;
    s->fwd_grid = std::max(1, fwd) * sms;
    s->bwd_grid = std::max(1, bwd) * sms;
    *out = s;
    return TRK_OK;
}

trk_status soft_launch(trk_tracker *t, const float *params, int lam, const uint32_t *mask, float sigma, float *loss,
                       float *grad, cudaStream_t st)
{
    if (lam == 0) return TRK_OK;
    SoftArgs a{};
    soft_shape(a, t);
    int slice = soft_fit(a, lam, true, kSoftBudget);
    SoftScratch *s = nullptr;
    trk_status r = soft_scratch(t, soft_layout(a, slice, true, nullptr), &s);
    if (r != TRK_OK) return r;
    slice = std::max(slice, soft_fit(a, lam, grad != nullptr, s->bytes));  // a loss alone needs less
    soft_layout(a, slice, grad != nullptr, static_cast<char *>(s->mem));
    a.fx = (float)t->cam.fx;
    a.fy = (float)t->cam.fy;
    a.cx = (float)(t->cam.cx256 / 256.0);
    a.cy = (float)(t->cam.cy256 / 256.0);
    a.z_near = (float)t->cam.z_near;
    a.guard = (float)t->cam.guard;
    a.sigma = sigma;
    a.verts = t->verts;
    a.tris = t->tris;
    a.mask = mask;
    for (int c0 = 0; c0 < lam; c0 += slice) {
        a.lam = std::min(slice, lam - c0);
        a.params = params + (size_t)c0 * a.d;
        a.loss = loss + c0;
        a.grad = grad ? grad + (size_t)c0 * a.d : nullptr;
        k_soft_fk<<<dim3(a.lam, a.nI), kSoftThreads, 0, st>>>(a);
        if (a.ngroups) {
            const int gpb = kSoftThreads / 32;
            k_soft_tris<<<dim3((a.ngroups + gpb - 1) / gpb, a.lam), kSoftThreads, a.nI * a.nF * 12 * sizeof(float),
                          st>>>(a);
        }
        const int pairs = (a.nby + 1) / 2 * a.nbx;
        k_soft_list<<<dim3((pairs + kSoftThreads - 1) / kSoftThreads, a.lam), kSoftThreads, 0, st>>>(a);
        k_soft_fwd<<<s->fwd_grid, 32 * kFwdWarps, 0, st>>>(a);
        if (grad) {
            if (a.ngroups) k_soft_bwd<<<s->bwd_grid, 32 * kBwdWarps, 0, st>>>(a);
            const int vpb = kSoftThreads * kRedVerts;
            k_soft_reduce<<<dim3(std::max(1, (a.V + vpb - 1) / vpb), a.lam * a.nI), kSoftThreads, 0, st>>>(a);
        }
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? TRK_OK : soft_fail(TRK_ECUDA, cudaGetErrorString(e));
}

}  // namespace

void trk::soft_free(trk_tracker *t)
{
    SoftScratch *s = static_cast<SoftScratch *>(t->soft);
    if (!s) return;
    cudaFree(s->mem);
    delete s;
    t->soft = nullptr;
}

void trk::refine_free(trk_cmaes *es)
{
    RefineBuf *r = static_cast<RefineBuf *>(es->refine);
    if (!r) return;
    cudaFree(r->P);
    cudaFree(r->g);
    cudaFree(r->m);
    cudaFree(r->v);
    cudaFree(r->ls);
    cudaFree(r->lh);
    cudaFree(r->order);
    cudaFree(r->picked);
    delete r;
    es->refine = nullptr;
}

extern "C" {

trk_status soft_eval(trk_tracker *t, const float *params_dev, int32_t lam, const uint32_t *mask_packed_dev,
                     float sigma, float *loss_dev, float *grad_dev, void *stream)
{
    if (!t) return soft_fail(TRK_EINVAL, "NULL tracker");
    if (lam < 0 || lam > TRK_MAX_LAMBDA) return soft_fail(TRK_EINVAL, "lam out of range");
    if (lam == 0) return TRK_OK;
    if (!params_dev || !mask_packed_dev || !loss_dev) return soft_fail(TRK_EINVAL, "NULL device pointer");
    if (!(sigma >= 0.05f && sigma <= 64.0f)) return soft_fail(TRK_EINVAL, "sigma must be in [0.05, 64] px");
    if (t->cam.W > 32767 || t->cam.H > 32767) return soft_fail(TRK_EINVAL, "image too large");
    return soft_launch(t, params_dev, lam, mask_packed_dev, sigma, loss_dev, grad_dev,
                       reinterpret_cast<cudaStream_t>(stream));
}

trk_status soft_refine(trk_cmaes *es, const uint32_t *mask_packed_dev, int32_t top_k, int32_t steps, float lr,
                       float sigma, float *pose_out_dev, int32_t *picked_host, void *stream)
{
    if (!es || !mask_packed_dev) return soft_fail(TRK_EINVAL, "NULL argument");
    if (top_k < 1 || top_k > 32 || top_k > es->lam) return soft_fail(TRK_EINVAL, "top_k must be 1..min(32, lam)");
    if (steps < 0 || steps > 1000) return soft_fail(TRK_EINVAL, "steps out of range");
    if (!(lr > 0.0f && lr < 10.0f)) return soft_fail(TRK_EINVAL, "lr out of range");
    if (!(sigma >= 0.05f && sigma <= 64.0f)) return soft_fail(TRK_EINVAL, "sigma must be in [0.05, 64] px");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    trk_tracker *t = es->t;
    RefineBuf *r = static_cast<RefineBuf *>(es->refine);
    if (!r) {
        r = new RefineBuf();
        const size_t n = (size_t)32 * es->d;
        cudaError_t e;
        if ((e = cudaMalloc(&r->P, sizeof(float) * n)) != cudaSuccess ||
            (e = cudaMalloc(&r->g, sizeof(float) * n)) != cudaSuccess ||
            (e = cudaMalloc(&r->m, sizeof(float) * n)) != cudaSuccess ||
            (e = cudaMalloc(&r->v, sizeof(float) * n)) != cudaSuccess ||
            (e = cudaMalloc(&r->ls, sizeof(float) * 32)) != cudaSuccess ||
            (e = cudaMalloc(&r->lh, sizeof(float) * 32)) != cudaSuccess ||
            (e = cudaMalloc(&r->order, sizeof(int) * 32)) != cudaSuccess ||
            (e = cudaMalloc(&r->picked, sizeof(int))) != cudaSuccess) {
            es->refine = r;
            refine_free(es);
            return soft_fail(e == cudaErrorMemoryAllocation ? TRK_ENOMEM : TRK_ECUDA, cudaGetErrorString(e));
        }
        r->cap = 32;
        es->refine = r;
    }
    const int d = es->d;
    k_refine_init<<<1, 128, 0, s>>>(es->params, es->loss, es->lam, d, top_k, r->P, r->m, r->v, r->order);
    for (int step = 1; step <= steps; ++step) {
        trk_status st = soft_launch(t, r->P, top_k, mask_packed_dev, sigma, r->ls, r->g, s);
        if (st != TRK_OK) return st;
        k_adam<<<(top_k * d + 127) / 128, 128, 0, s>>>(r->P, r->g, r->m, r->v, es->k, top_k, d, lr, 0.9f, 0.999f,
                                                       1e-8f, step);
    }
    // fitness (binary silhouette, the tracker's loss) of the refined candidates
    EvalArgs a{};
    a.ch = t->ch;
    a.cam = t->cam;
    apply_mesh(a, t);
    a.params = r->P;
    a.d = d;
    a.lam = top_k;
    a.mask = mask_packed_dev;
    a.snap = t->snap;
    a.loss = r->lh;
    a.loss_kind = t->cfg.loss_kind;
    a.lambda_app = t->cfg.lambda_app;
    a.cull = t->cfg.cull_backfaces;
    apply_keypoints(a, t);
    cudaError_t e = launch_eval(a, t->lc, s);
    if (e != cudaSuccess) return soft_fail(TRK_ECUDA, cudaGetErrorString(e));
    k_refine_pick<<<1, 32, 0, s>>>(r->P, r->lh, top_k, d, es->st, pose_out_dev, r->picked);
    if ((e = cudaGetLastError()) != cudaSuccess) return soft_fail(TRK_ECUDA, cudaGetErrorString(e));
    if (picked_host) {
        if ((e = cudaMemcpyAsync(picked_host, r->picked, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
            (e = cudaStreamSynchronize(s)) != cudaSuccess)
            return soft_fail(TRK_ECUDA, cudaGetErrorString(e));
    }
    return TRK_OK;
}

}  // extern "C"
