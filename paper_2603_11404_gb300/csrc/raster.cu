// Fitness of a CMA-ES population in one launch (arXiv 2603.11404, Sec. III-A.2):
//   S = R(K(Pi(T_r^c T_m^r(q) v_m))),  counts (s, I, m) of S against M_ref,
//   loss of Eq. render_loss / the 1 - IoU mask error of Sec. IV-B.
//
// Launch shape: one thread-block cluster of `cluster` CTAs per candidate.
//   prologue every CTA of the cluster (in the fused CMA-ES mode) samples the
//            candidate and composes its link transforms in double-float
//            arithmetic (redundantly: no CTA waits for another).
//   phase 1  every CTA projects its share of the vertices in compensated FP32
//            (double-float, error-free TwoSum/TwoProd), snapping them to 1/256 px
//            with round-half-even; the snapped vertices go to an L2-resident
//            scratch array.
//   phase 2  after a cluster barrier the warps of all CTAs take chunks of 32
//            primitive records (edge-sharing triangle pairs, drawn as convex
//            quadrilaterals where the projected corners allow, else as their
//            triangles) from a counter in CTA 0's shared memory until none
//            are left.  Primitives with a pixel centre in their box (on a
//            closed mesh the front faces alone) enter the warp's queue, and a
//            full queue is drawn a row of pixels per lane with int32 edge
//            functions; larger ones are deferred and, after a second cluster
//            barrier, drawn by the warps of the whole cluster, a row per lane
//            from its edges' crossings.  Coverage is OR-ed into the CTA's own
//            full-image bitmap in shared memory.
//   phase 3  after a further cluster barrier CTA r ORs band r of all the
//            cluster's bitmaps through distributed shared memory, ANDs with
//            the observed mask, popcounts, and the cluster's counts meet in
//            CTA 0, which writes counts and loss.
// No silhouette image is written to global memory.
#include <cooperative_groups.h>

#include "raster_dev.cuh"

namespace cg = cooperative_groups;

namespace trk {

// Front of the dynamic shared memory: the composition's scratch and, once the
// frames are composed, the warps' drawing queues (room for 8 warps at least).
constexpr int kQueueEntryBytes = 40;  // an entry of draw_rows' table; a queued primitive takes 32

__host__ __device__ inline size_t front_smem_bytes(int n_inst, int qcap, int threads)
{
    const size_t warps = threads > 256 ? threads / 32 : 8;
    const size_t scr = (size_t)n_inst * kComposeScratch * sizeof(float2), q = warps * qcap * kQueueEntryBytes;
    return scr > q ? scr : q;
}

constexpr int kAccWords = 12;  // counters behind the deferred list (see eval_candidate)

// Projected keypoints of given states (synthetic detections, diagnostics):
// one warp per state composes its frames and writes (u, v) of both keypoints
// of every instrument.
__global__ void k_project_keypoints(EvalArgs a, const float *states, int n, float *out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int nI = a.ch.n_inst, nF = a.ch.n_frames;
    float2 *scr = reinterpret_cast<float2 *>(smem);
    float *sM = reinterpret_cast<float *>(scr + nI * kComposeScratch);
    const int st = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (st >= n) return;
    if (warp < nI)
        compose_frames_warp(a.ch, a.cam, states + (size_t)st * a.d + 9 * warp, sM + warp * nF * 24,
                            scr + warp * kComposeScratch, lane);
    __syncthreads();
    if (threadIdx.x < 2 * nI) {
        const int b = threadIdx.x >> 1, k = threadIdx.x & 1;
        const float2 p = project_keypoint(sM + (b * nF + a.kp_frame[k]) * 24, a.kp_pt[k], a.cam);
        out[((size_t)st * nI + b) * 4 + 2 * k] = p.x;
        out[((size_t)st * nI + b) * 4 + 2 * k + 1] = p.y;
    }
}

cudaError_t launch_project_keypoints(const EvalArgs &a, const float *states, int n, float *out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const size_t smem = (size_t)a.ch.n_inst * (kComposeScratch * sizeof(float2) + a.ch.n_frames * 24 * sizeof(float));
    k_project_keypoints<<<n, 32 * a.ch.n_inst, smem, s>>>(a, states, n, out);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// The fused fitness kernel.
// ----------------------------------------------------------------------------

// One candidate c of one evaluation (all CTAs of the cluster call it together).
// mask_override replaces a.mask when not NULL (batched launches).  A non-zero
// tell_ctas is the number of CTAs that evaluate a's population in this launch:
// the last of them to finish runs the CMA-ES update (and, when a.cma_finish is
// set, the frame epilogue).
// Consecutive fused generations are launched with programmatic stream
// serialisation (see griddep_wait).
// Triangle t's vertex indices.  kChecked (meshes in the caller's device memory,
// which the host cannot validate): an index outside [0, V) marks the triangle
// bad (w = 1) and points it at vertex 0, so nothing outside the candidate's
// vertices is read; gather3 then flags it, and it is culled.
template <bool kChecked>
__device__ __forceinline__ int4 load_tri(const EvalArgs &a, int t)
{
    const int b = t >= a.T;  // instrument (at most 2): no division
    int4 tri = a.tris[t - b * a.T];
    if (kChecked) {
        const bool ok = (unsigned)tri.x < (unsigned)a.V && (unsigned)tri.y < (unsigned)a.V &&
                        (unsigned)tri.z < (unsigned)a.V;
        tri = ok ? make_int4(tri.x, tri.y, tri.z, 0) : make_int4(0, 0, 0, 1);
    }
    return tri;
}

// The three snapped vertices of a loaded triangle (written by other CTAs of
// the cluster: read through L2).
template <bool kChecked>
__device__ __forceinline__ void gather3(const int2 *sv, int4 tri, int2 &v0, int2 &v1, int2 &v2)
{
    v0 = __ldcg(sv + tri.x);
    v1 = __ldcg(sv + tri.y);
    v2 = __ldcg(sv + tri.z);
    if (kChecked && tri.w) v0.x = kSnapFlag;
}

// Chunk tickets of phase 2: lane 0 takes the next chunk from the counter in
// CTA 0's shared memory and broadcasts it.
__device__ __forceinline__ int chunk_ticket(int *ctr, int lane)
{
    int v = 0;
    if (lane == 0) v = atomicAdd(ctr, 1);
    return __shfl_sync(0xffffffffu, v, 0);
}

__device__ __forceinline__ bool small_box(int spanx, int spany) { return spanx < 32 * 256 && spany < 64 * 256; }

// One triangle of phase 2: drawn by this lane when small, otherwise deferred to
// a whole warp through the CTA's list (entry `ent`).  Returns 1 when the
// triangle is culled for a flagged vertex.
__device__ __forceinline__ int draw_one_tri(int2 v0, int2 v1, int2 v2, int ent, const EvalArgs &a, int cull,
                                            uint32_t *bm, int *big, int *sacc)
{
    TriSetup t;
    const int st = tri_setup(v0, v1, v2, a.cam.W, a.cam.H, cull, t);
    if (st == 1) {
        if (small_box(t.spanx, t.spany)) {
            raster_small(t, bm, a.cam.Wq);
        } else {
            // larger triangles wait for a whole warp.  If the list is full,
            // every large triangle is drawn again after the loop (raster code
            // here would make it spill)
            const int slot = atomicAdd(&sacc[4], 1);
            if (slot < kBigListCap) big[slot] = ent;
            else sacc[6] = 1;
        }
    }
    return st == 2;
}

// Primitive t's record and snapped corners (written by other CTAs of the
// cluster: read through L2).  A single triangle has w = -1 and no 4th corner.
__device__ __forceinline__ int4 load_prim(const EvalArgs &a, int t)
{
    const int b = t >= a.P;  // instrument (at most 2): no division
    return a.prims[t - b * a.P];
}

__device__ __forceinline__ void gather_prim(const EvalArgs &a, const int2 *snapc0, int t, int4 p, int2 &v0, int2 &v1,
                                            int2 &v2, int2 &v3)
{
    const int2 *sv = snapc0 + (t >= a.P) * a.V;
    v0 = __ldcg(sv + p.x);
    v1 = __ldcg(sv + p.y);
    v2 = __ldcg(sv + p.z);
    if (p.w >= 0) v3 = __ldcg(sv + p.w);
}

// A large entry waits for the end of the loop, unless none of its triangles is
// to be drawn.  If the list is full, every large primitive is drawn again after
// the loop (raster code here would make it spill).
__device__ __forceinline__ void defer_large(int t, const PrimEntry &e, const EvalArgs &a, int cull, int *big, int *sacc)
{
    const int W = a.cam.W, H = a.cam.H;
    TriSetup ts;
    if (tri_setup(e.c0, e.c1, e.c2, W, H, cull, ts) != 1 &&
        (e.c3.x == kSnapFlag || tri_setup(e.c0, e.c2, e.c3, W, H, cull, ts) != 1))
        return;
    const int slot = atomicAdd(&sacc[4], 1);
    if (slot < kBigListCap) big[slot] = 4 * t + e.part;
    else sacc[6] = 1;
}

// Phase 2 over the tracker's primitive list (quadrilateral pairs and single
// triangles, prims[] of EvalArgs).  A warp takes a chunk of 32 primitives
// (one per lane) from the cluster's counter and takes the next chunk's ticket
// while it sets the current one up: a warp holds at most one chunk beyond the
// one it works on, so the warps of a cluster run out of work together.
// Set-up and drawing are apart: of the 32 primitives of a chunk five to ten are
// front faces with a pixel centre in their box (640x512, 20k triangles).  The
// warp queues those (EvalArgs::qcap entries in shared memory) and takes a full
// queue at a time through the convexity test, the edge set-up and the drawing.
// Deferred-list entries are 4 * primitive + part: part 0 the whole
// quadrilateral (its two triangles), 1 its first triangle (a, b, c), 2 its
// second (a, c, d); they are drawn after the cluster barrier that follows,
// shared out over the whole cluster (in eval_candidate).  `cull` leaves out
// back faces.  Returns this thread's count of triangles culled for a flagged
// vertex.
__device__ __forceinline__ int draw_prims(const EvalArgs &a, int cull, cg::cluster_group &cluster, const int2 *snapc0,
                                          uint32_t *bm, int *big, int *sacc, int4 *queue, int lane, int warp, int nwarp)
{
    const int W = a.cam.W, H = a.cam.H, Wq = a.cam.Wq;
    const int NP = a.ch.n_inst * a.P, cap = a.qcap;
    int culled = 0;
    int *ctr = cluster.map_shared_rank(&sacc[5], 0);
    int cur = chunk_ticket(ctr, lane), qn = 0;
    for (;;) {
        PrimEntry e;
        bool live = false;
        const bool last = cur * 32 >= NP;  // tickets of one warp increase: once past the end, done
        if (!last) {
            int tk = 0;
            if (lane == 0) tk = atomicAdd(ctr, 1);  // the next chunk, read after this one's set-up
            const int t = cur * 32 + lane;
            if (t < NP) {
                const int4 p = load_prim(a, t);
                int2 v0, v1, v2, v3 = make_int2(0, 0);
                gather_prim(a, snapc0, t, p, v0, v1, v2, v3);
                if (make_entry(v0, v1, v2, v3, p.w >= 0, culled, e)) {
                    const int size = entry_size(e, W, H);
                    live = size == 1 && !(cull && back_small(e));
                    if (size == 2) defer_large(t, e, a, cull, big, sacc);
                }
            }
            cur = __shfl_sync(0xffffffffu, tk, 0);
        }
        const unsigned m = __ballot_sync(0xffffffffu, live);
        int pos = qn + __popc(m & ((1u << lane) - 1u));
        qn += __popc(m);
        for (;;) {  // enter what fits, draw the queue when it is full
            if (live && pos < cap) {
                queue[pos] = make_int4(e.c0.x, e.c0.y, e.c1.x, e.c1.y);
                queue[cap + pos] = make_int4(e.c2.x, e.c2.y, e.c3.x, e.c3.y);
                live = false;
            }
            if (qn < cap && !(last && qn > 0)) break;
            __syncwarp();
            const bool on = lane < min(qn, cap);
            int4 p = make_int4(0, 0, 0, 0), q = p;
            if (on) {
                p = queue[lane];
                q = queue[cap + lane];
            }
            __syncwarp();  // the queue's memory becomes the row table
            draw_rows(on, make_int2(p.x, p.y), make_int2(p.z, p.w), make_int2(q.x, q.y), make_int2(q.z, q.w), W, H, cull,
                      bm, Wq, queue, cap, lane);
            qn = max(qn - cap, 0);
            pos -= cap;
        }
        if (last) break;
    }
    __syncthreads();
    if (sacc[6]) {
        // the list overflowed: every large primitive of the candidate (drawing
        // twice is harmless under the union); a primitive counts as large
        // exactly as in the loop above
        for (int base = warp * 32; base < NP; base += nwarp * 32) {
            const int tt = base + lane;
            PrimEntry e;
            bool large = false;
            if (tt < NP) {
                const int4 p = load_prim(a, tt);
                int2 u0, u1, u2, u3 = make_int2(0, 0);
                gather_prim(a, snapc0, tt, p, u0, u1, u2, u3);
                int dummy = 0;
                large = make_entry(u0, u1, u2, u3, p.w >= 0, dummy, e) && entry_size(e, W, H) == 2;
            }
            const unsigned m = __ballot_sync(0xffffffffu, large);
            const int pos = __popc(m & ((1u << lane) - 1u));
            for (int b = 0; b < __popc(m); b += cap)
                draw_rows_large(large && pos >= b && pos < b + cap, e.c0, e.c1, e.c2, e.c3, W, H, cull, bm, Wq, queue, cap,
                                lane);
        }
    }
    return culled;
}

// Phase 2 over plain triangles (tris[] of EvalArgs; the index-checked launch on
// meshes in caller memory).  Deferred-list entries are triangle indices.
template <bool kChecked>
__device__ __forceinline__ int draw_tris(const EvalArgs &a, cg::cluster_group &cluster, const int2 *snapc, uint32_t *bm,
                                      int *big, int *sacc, int lane, int warp, int nwarp)
{
    const int W = a.cam.W, H = a.cam.H, Wq = a.cam.Wq;
    int culled = 0;
    const int NT = a.ch.n_inst * a.T;
    int *ctr = cluster.map_shared_rank(&sacc[5], 0);
    int cur = chunk_ticket(ctr, lane), nx1 = chunk_ticket(ctr, lane), nx2 = chunk_ticket(ctr, lane);
    int t0 = cur * 32 + lane, t1 = nx1 * 32 + lane;
    int4 tri1 = make_int4(0, 0, 0, 0);
    int b1 = 0;
    int2 v0 = make_int2(0, 0), v1 = v0, v2 = v0;
    if (t0 < NT) {
        const int b0 = t0 >= a.T;  // instrument (at most 2): no division
        gather3<kChecked>(snapc + b0 * a.V, load_tri<kChecked>(a, t0), v0, v1, v2);
    }
    if (t1 < NT) {
        b1 = t1 >= a.T;
        tri1 = load_tri<kChecked>(a, t1);
    }
    while (cur * 32 < NT) {
        const int nx3 = chunk_ticket(ctr, lane);
        int2 w0 = make_int2(0, 0), w1 = w0, w2 = w0;
        if (t1 < NT) gather3<kChecked>(snapc + b1 * a.V, tri1, w0, w1, w2);
        const int t2 = nx2 * 32 + lane;
        int4 tri2 = make_int4(0, 0, 0, 0);
        int b2 = 0;
        if (t2 < NT) {
            b2 = t2 >= a.T;
            tri2 = load_tri<kChecked>(a, t2);
        }
        if (t0 < NT) culled += draw_one_tri(v0, v1, v2, t0, a, a.cull, bm, big, sacc);
        cur = nx1;
        t0 = t1;
        v0 = w0;
        v1 = w1;
        v2 = w2;
        nx1 = nx2;
        t1 = t2;
        tri1 = tri2;
        b1 = b2;
        nx2 = nx3;
    }
    __syncthreads();
    const int nbig = min(sacc[4], kBigListCap);
    for (int e = warp; e < nbig; e += nwarp) {
        int tt = big[e];
        int b = tt >= a.T;
        int2 u0, u1, u2;
        gather3<kChecked>(snapc + b * a.V, load_tri<kChecked>(a, tt), u0, u1, u2);
        TriSetup t;
        tri_setup(u0, u1, u2, W, H, a.cull, t);
        raster_warp(t, bm, Wq, lane);
    }
    if (sacc[6]) {  // the list overflowed: every large triangle of the candidate, a warp each (drawing twice is harmless)
        for (int base = warp * 32; base < NT; base += nwarp * 32) {
            const int tt = base + lane;
            bool large = false;
            TriSetup t;
            if (tt < NT) {
                const int b = tt >= a.T;
                int2 u0, u1, u2;
                gather3<kChecked>(snapc + b * a.V, load_tri<kChecked>(a, tt), u0, u1, u2);
                large = tri_setup(u0, u1, u2, W, H, a.cull, t) == 1 && !small_box(t.spanx, t.spany);
            }
            for (unsigned mm = __ballot_sync(0xffffffffu, large); mm; mm &= mm - 1) {
                const int src = __ffs(mm) - 1, tu = __shfl_sync(0xffffffffu, tt, src);
                const int b = tu >= a.T;
                int2 u0, u1, u2;
                gather3<kChecked>(snapc + b * a.V, load_tri<kChecked>(a, tu), u0, u1, u2);
                TriSetup u;
                tri_setup(u0, u1, u2, W, H, a.cull, u);
                raster_warp(u, bm, Wq, lane);
            }
        }
    }
    return culled;
}

template <bool kChecked = false, bool kQuads = true>
__device__ __forceinline__ void eval_candidate(const EvalArgs &a, int c, const uint32_t *mask_override,
                                               unsigned tell_ctas, bool dependent_launch)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int K = (int)cluster.num_blocks();
    const uint32_t *maskp = mask_override ? mask_override : a.mask;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
    const int nI = a.ch.n_inst, nF = a.ch.n_frames;
    const int H = a.cam.H, Wq = a.cam.Wq;
    const int nwords = H * Wq;

    extern __shared__ __align__(16) unsigned char smem[];
    float2 *scr = reinterpret_cast<float2 *>(smem);                           // [nI*kComposeScratch]
    int4 *queues = reinterpret_cast<int4 *>(smem);                            // [nwarp][qcap entries]: phase 2, over scr
    uint32_t *bm = reinterpret_cast<uint32_t *>(smem + front_smem_bytes(nI, a.qcap, blockDim.x));  // [H*Wq]
    float *sM = reinterpret_cast<float *>(bm + ((nwords + 3) & ~3));          // [nI*nF*24]
    int *big = reinterpret_cast<int *>(sM + nI * nF * 24);                    // [kBigListCap]
    // [kAccWords]: s I m culled, big-list count, chunk ticket counter, big-list
    // overflow, deferred-entry ticket counter, a vertex of this CTA is flagged
    int *sacc = big + kBigListCap;
    __shared__ int red[4][32];
    __shared__ float s_par[kMaxD];
    __shared__ float2 s_z[kMaxD];
    __shared__ int s_last;

    const bool two_warps = nwarp > 2 * nI;  // an instrument's frames are composed by two warps
    {  // the warps that do not compose frames clear the bitmap (16-byte stores)
        const int c0 = two_warps ? 64 * nI : nwarp > nI ? 32 * nI : 0;
        uint4 *bm4 = reinterpret_cast<uint4 *>(bm);
        for (int w = tid - c0; w >= 0 && w < (nwords + 3) >> 2; w += nthr - c0) bm4[w] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (tid < kAccWords) sacc[tid] = 0;
    // everything above touches only this CTA's shared memory; from here on the
    // launch reads what the previous generation wrote
    if (dependent_launch) griddep_wait();
    // ---- prologue: every CTA samples the candidate (fused CMA-ES mode; the
    //      draws are the same in every CTA and CTA 0 stores them) and composes
    //      its frames in double-float, so no CTA waits for another ----
    {
        const float *par = a.params + (size_t)c * a.d;
        if (a.cma_st) {
            if (warp == 0) {
                const bool owner = rank == 0;
                cma_sample_warp(*a.cma_k, a.cma_st, c, nullptr, owner ? a.cma_y : nullptr,
                                owner ? a.cma_z : nullptr, owner ? const_cast<float *>(a.params) : nullptr, s_par,
                                s_z, lane);
            }
            __syncthreads();
            par = s_par;
        }
        if (two_warps) {
            if (warp < nI) compose_joints(a.ch, par + 9 * warp, scr + warp * kComposeScratch, lane);
            else if (warp < 2 * nI) compose_pose(a.ch, a.cam, par + 9 * (warp - nI), scr + (warp - nI) * kComposeScratch, lane);
            __syncthreads();
            if (warp < nI) compose_chain(a.ch, sM + warp * nF * 24, scr + warp * kComposeScratch, lane);
        } else if (warp < nI) {
            compose_frames_warp(a.ch, a.cam, par + 9 * warp, sM + warp * nF * 24, scr + warp * kComposeScratch,
                                lane);
        }
        if (rank == 0 && warp == nwarp - 1) check_state_finite(par, a.d, a.err, lane);
    }
    __syncthreads();

    // ---- phase 1: project and snap this CTA's share of the vertices ----
    int2 *snapc = a.snap + (size_t)c * nI * a.V;
    const int NV = nI * a.V;
    for (int idx = rank * nthr + tid; idx < NV; idx += K * nthr) {
        const int b = idx >= a.V;  // instrument (at most 2): no division
        const float4 p = a.verts[idx - b * a.V];
        float2 uv = make_float2(0.0f, 0.0f);
        int2 o = make_int2(kSnapFlag, kSnapFlag);
        const int f = (int)p.w;
        if (!kChecked || ((unsigned)f < (unsigned)nF && (float)f == p.w))  // else: a frame index out of range
            o = project_vertex(p, sM + (b * nF + f) * 24, a.cam, uv);
        snapc[idx] = o;
        if (a.snap_dbg) a.snap_dbg[(size_t)c * NV + idx] = o;
        if (a.uv_dbg) a.uv_dbg[(size_t)c * NV + idx] = uv;
        if (o.x == kSnapFlag) sacc[8] = 1;
    }
    cluster.sync();  // arrive.release / wait.acquire: the snapped vertices are visible cluster-wide

    // ---- phase 2: primitives -> this CTA's bitmap.  Warps of the whole cluster
    //      take chunks of 32 primitives (one per lane) from a counter in CTA 0's
    //      shared memory, so the cluster finishes together whatever they cost;
    //      the bitmaps are OR-ed in phase 3, so which CTA draws a primitive does
    //      not change the result ----
    // A closed mesh without a flagged vertex is drawn by its front faces
    // alone: the edges of its triangles cancel in pairs, so the triangles that
    // cover a pixel centre (see the quadrilateral rule: no centre lies on an
    // edge) have as many positive as negative orientations among them -- a
    // pixel that any triangle covers, some front face covers.  A flagged
    // vertex drops triangles and opens the surface.
    int cull = a.cull;
    if (kQuads && a.closed)
        cull |= !__any_sync(0xffffffffu, lane < K && *cluster.map_shared_rank(&sacc[8], lane < K ? lane : 0) != 0);
    int culled = kQuads ? draw_prims(a, cull, cluster, snapc, bm, big, sacc, queues + a.qcap * kQueueEntryBytes / 16 * warp, lane,
                                                       warp, nwarp)
                        : draw_tris<kChecked>(a, cluster, snapc, bm, big, sacc, lane, warp, nwarp);
    cluster.sync();
    if (kQuads) {
        // the large primitives deferred by every CTA of the cluster, shared out
        // over all its warps: the tip of a coarse mesh close to the camera lands
        // in a few chunks, and a CTA drawing its own list alone would hold the
        // whole cluster up.  Entry e of the cluster is entry e - start(r) of
        // CTA r's list (lists read through DSMEM, complete at the barrier above)
        const int cnt = lane < K ? min(*cluster.map_shared_rank(&sacc[4], lane), kBigListCap) : 0;
        int incl = cnt;
        for (int o = 1; o < 8; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 7);
        if (total > 0) {  // the same in every CTA: the barrier below is uniform
            // a ticket stands for `per` entries: one while there are warps enough
            // (its rows go to the lanes), more when the list is long
            int *ctr = cluster.map_shared_rank(&sacc[7], 0);
            const int per = min(a.qcap, (total + K * nwarp - 1) / (K * nwarp));
            for (int e0 = chunk_ticket(ctr, lane) * per; e0 < total; e0 = chunk_ticket(ctr, lane) * per) {
                const int e = e0 + lane;
                int r = 0, start = 0;
                for (int q = 0; q < K; ++q) {
                    const int v = __shfl_sync(0xffffffffu, incl, q);
                    if (v <= e) {
                        r = q + 1;
                        start = v;
                    }
                }
                const bool live = lane < per && e < total;
                int2 c0 = make_int2(0, 0), c1 = c0, c2 = c0, c3 = make_int2(kSnapFlag, kSnapFlag);
                if (live) {
                    const int ent = cluster.map_shared_rank(big, r)[e - start], t = ent >> 2, part = ent & 3;
                    const int b = t >= a.P;
                    const int4 p = a.prims[t - b * a.P];
                    const int2 *sv = snapc + b * a.V;
                    c0 = __ldcg(sv + p.x);
                    c1 = __ldcg(sv + (part == 2 ? p.z : p.y));
                    c2 = __ldcg(sv + (part == 2 ? p.w : p.z));
                    if (part == 0) c3 = __ldcg(sv + p.w);
                }
                draw_rows_large(live, c0, c1, c2, c3, a.cam.W, H, cull, bm, Wq, queues + a.qcap * kQueueEntryBytes / 16 * warp,
                                a.qcap, lane);
            }
            cluster.sync();  // every deferred primitive drawn before the bitmaps are read
        }
    }

    // ---- phase 3: OR the cluster's bitmaps over this CTA's band, count ----
    const int per = (nwords + K - 1) / K;
    const int w0 = rank * per, w1 = min(nwords, w0 + per);
    const uint32_t *rbm[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) rbm[q] = cluster.map_shared_rank(bm, q < K ? q : 0);
    int s = 0, I = 0, m = 0;
    for (int w = w0 + tid; w < w1; w += nthr) {
        uint32_t part[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) part[q] = (q < K) ? rbm[q][w] : 0u;
        uint32_t M = maskp[w];
        uint32_t S = 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) S |= part[q];
        s += __popc(S);
        I += __popc(S & M);
        m += __popc(M);
        if (a.silhouette) a.silhouette[w] = S;
    }
    for (int o = 16; o; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        I += __shfl_xor_sync(0xffffffffu, I, o);
        m += __shfl_xor_sync(0xffffffffu, m, o);
        culled += __shfl_xor_sync(0xffffffffu, culled, o);
    }
    if (lane == 0) {
        red[0][warp] = s;
        red[1][warp] = I;
        red[2][warp] = m;
        red[3][warp] = culled;
    }
    __syncthreads();
    if (tid < 4) {
        int acc = 0;
        for (int w = 0; w < nwarp; ++w) acc += red[tid][w];
        atomicAdd(cluster.map_shared_rank(&sacc[tid], 0), acc);
    }
    cluster.sync();
    if (rank == 0 && tid == 0) {
        int S_ = sacc[0], I_ = sacc[1], M_ = sacc[2], C_ = sacc[3];
        if (a.counts) {
            a.counts[4 * c + 0] = S_;
            a.counts[4 * c + 1] = I_;
            a.counts[4 * c + 2] = M_;
            a.counts[4 * c + 3] = C_;
        }
        if (a.loss) {
            int x = S_ + M_ - 2 * I_;
            float L;
            if (a.loss_kind == TRK_LOSS_ONE_MINUS_IOU) {
                int U = S_ + M_ - I_;
                L = (U > 0) ? __fsub_rn(1.0f, __fdiv_rn((float)I_, (float)U)) : 0.0f;
            } else if (a.loss_kind == TRK_LOSS_MSE_APP) {
                L = __fadd_rn((float)x, __fmul_rn(a.lambda_app, (float)abs(S_ - M_)));
            } else {
                L = (float)x;
            }
            if (a.kp_obs && a.kp_lambda != 0.0f) L = __fadd_rn(L, keypoint_loss(a, sM));
            a.loss[c] = L;
        }
    }
    if (a.cma_st && tell_ctas) {  // the last CTA to finish updates the search distribution
        if (tid == 0) {
            __threadfence();
            unsigned ticket = atomicAdd(a.cma_done, 1u);
            s_last = (ticket == tell_ctas - 1);
        }
        __syncthreads();
        if (s_last) {
            __threadfence();
            TellSmem &S = *reinterpret_cast<TellSmem *>(smem);  // the cluster no longer reads this CTA's smem
            // a frame's last generation leaves out the square roots: the next
            // frame restarts from C = I (the host runs them if it does not)
            cma_tell_block(*a.cma_k, a.cma_st, a.cma_y, a.params, a.loss, S, tid, nthr, !a.cma_finish);
            __syncthreads();
            if (a.cma_finish) cma_finish_frame(*a.cma_k, a.cma_st, a.cma_pose_out, tid, nthr);
            if (tid == 0) *a.cma_done = 0u;
        }
    }
}

__global__ void __launch_bounds__(256, 4) k_eval(EvalArgs a)
{
    griddep_launch_dependents();
    eval_candidate<>(a, blockIdx.y, nullptr, gridDim.x * gridDim.y, true);
}

// The same in CTAs of up to 1024 threads (see eval_wide_threads).
__global__ void __launch_bounds__(1024, 1) k_eval_wide(EvalArgs a)
{
    griddep_launch_dependents();
    eval_candidate<>(a, blockIdx.y, nullptr, gridDim.x * gridDim.y, true);
}

// The same with index checks: meshes in the caller's device memory
// (eval_population_noalloc), whose indices the host cannot validate.
__global__ void __launch_bounds__(256, 4) k_eval_checked(EvalArgs a)
{
    eval_candidate<true, false>(a, blockIdx.y, nullptr, 0u, false);
}

// Persistent batched evaluation: a fixed grid of clusters pulls (instance,
// candidate) items from a queue (largest first) until it is empty.  CTA 0 of
// each cluster takes the ticket and the others read it through DSMEM, so the
// cluster stays in lockstep.  kTell (serving ticks): tell_last holds one flag
// per instance (1 for a frame's last generation) and the last CTA of each
// instance's items runs that instance's CMA-ES update, as k_eval does for one
// instance; items and flags sit in mapped pinned host memory that the host
// rewrites between ticks (read with ld.cv, never from a cached line), and the
// cluster that draws the launch's last ticket leaves the queue counter at zero
// for the next tick.  Without kTell the updates are a separate launch.
// Four CTAs to an SM with the updates, at 64 registers: eight streams at 640x512
// take 7.45 ms for 32 frames, with three 7.90; a batch's frames of one CTA per
// candidate are no faster with four (7.3 against 6.8 ms).
template <bool kTell, bool kWide>
__device__ __forceinline__ void eval_batch_body(const EvalArgs *descs, const uint32_t *const *masks, const int2 *items,
                                                int n_items, unsigned *next_item, const int *tell_last, int wide_qcap)
{
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ int s_item;
    __shared__ int s_tick[3];  // kTell: the item and its instance's flag, read once by CTA 0's thread 0
    __shared__ __align__(16) EvalArgs s_args;  // this item's descriptor, read from shared memory
    for (;;) {
        if (cluster.block_rank() == 0 && threadIdx.x == 0) {
            s_item = (int)atomicAdd(next_item, 1u);
            if (kTell && s_item < n_items) {
                const int2 v = __ldcv(items + s_item);
                s_tick[0] = v.x;
                s_tick[1] = v.y;
                s_tick[2] = __ldcv(tell_last + v.x);
            }
        }
        cluster.sync();
        const int it = *cluster.map_shared_rank(&s_item, 0);
        int2 ic = make_int2(0, 0);
        int last = 0;
        if (kTell && it < n_items) {
            const int *t0 = cluster.map_shared_rank(s_tick, 0);
            ic = make_int2(t0[0], t0[1]);
            last = t0[2];
        }
        cluster.sync();  // every CTA has its ticket before CTA 0 takes the next
        if (it >= n_items) {
            // every cluster draws exactly one ticket past the items: the last of
            // them is the launch's last atomic on the counter
            if (kTell && cluster.block_rank() == 0 && threadIdx.x == 0 && it == n_items + (int)gridDim.y - 1)
                *next_item = 0u;
            break;
        }
        if (!kTell) ic = items[it];
        const int4 *src = reinterpret_cast<const int4 *>(descs + ic.x);
        int4 *dst = reinterpret_cast<int4 *>(&s_args);
        for (int i = threadIdx.x; i < (int)(sizeof(EvalArgs) / 16); i += blockDim.x) dst[i] = src[i];
        __syncthreads();
        unsigned tell = 0;
        if (kTell) {
            if (threadIdx.x == 0) s_args.cma_finish = last;
            __syncthreads();
            tell = (unsigned)s_args.lam * gridDim.x;  // every CTA of every candidate of the instance
        }
        if (kWide) {  // the descriptor's queues are sized for 256 threads
            if (threadIdx.x == 0) s_args.qcap = wide_qcap;
            __syncthreads();
        }
        eval_candidate<>(s_args, ic.y, masks ? masks[ic.x] : nullptr, tell, false);
    }
}

template <bool kTell>
__global__ void __launch_bounds__(256, kTell ? 4 : 3)
    k_eval_batch(const EvalArgs *descs, const uint32_t *const *masks, const int2 *items, int n_items,
                 unsigned *next_item, const int *tell_last)
{
    eval_batch_body<kTell, false>(descs, masks, items, n_items, next_item, tell_last, 0);
}

__global__ void __launch_bounds__(1024, 1) k_eval_batch_wide(const EvalArgs *descs, const uint32_t *const *masks,
                                                             const int2 *items, int n_items, unsigned *next_item,
                                                             int qcap)
{
    eval_batch_body<false, true>(descs, masks, items, n_items, next_item, nullptr, qcap);
}

cudaError_t launch_eval_batch(const EvalArgs *descs_dev, const uint32_t *const *masks_dev, const int2 *items_dev,
                              int n_items, unsigned *next_item_dev, const LaunchCfg &cfg, int n_clusters,
                              cudaStream_t s, const int *tell_last_dev)
{
    if (n_items == 0) return cudaSuccess;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cfg.cluster, n_clusters, 1);
    lc.blockDim = dim3(cfg.threads, 1, 1);
    lc.dynamicSmemBytes = cfg.smem;
    lc.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cfg.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    if (cfg.threads > 256)  // batches only: the updates are a launch of their own
        return cudaLaunchKernelEx(&lc, k_eval_batch_wide, descs_dev, masks_dev, items_dev, n_items, next_item_dev,
                                  cfg.qcap);
    return tell_last_dev ? cudaLaunchKernelEx(&lc, k_eval_batch<true>, descs_dev, masks_dev, items_dev, n_items,
                                              next_item_dev, tell_last_dev)
                         : cudaLaunchKernelEx(&lc, k_eval_batch<false>, descs_dev, masks_dev, items_dev, n_items,
                                              next_item_dev, tell_last_dev);
}

cudaError_t prepare_eval_batch(size_t smem, int cluster, int threads, bool tell, int *max_clusters)
{
    const bool wide = threads > 256;
    const cudaError_t e = ensure_smem_attr(wide   ? (const void *)k_eval_batch_wide
                                           : tell ? (const void *)k_eval_batch<true>
                                                  : (const void *)k_eval_batch<false>,
                                           smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cluster, 1, 1);
    lc.blockDim = dim3(threads, 1, 1);
    lc.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return wide   ? cudaOccupancyMaxActiveClusters(max_clusters, k_eval_batch_wide, &lc)
           : tell ? cudaOccupancyMaxActiveClusters(max_clusters, k_eval_batch<true>, &lc)
                  : cudaOccupancyMaxActiveClusters(max_clusters, k_eval_batch<false>, &lc);
}

size_t tell_smem_bytes() { return sizeof(TellSmem); }

// Shared memory of a CTA behind its front.
static size_t eval_rest_bytes(const ChainDev &ch, const CamDev &cam)
{
    const size_t nwords = (size_t)cam.H * cam.Wq;
    return ((nwords + 3) & ~(size_t)3) * 4 + (size_t)ch.n_inst * ch.n_frames * 24 * 4 + (size_t)kBigListCap * 4 +
           kAccWords * 4;
}

size_t eval_smem_bytes(const EvalArgs &a, int threads, size_t reserve)
{
    return front_smem_bytes(a.ch.n_inst, eval_queue_cap(a.ch, a.cam, threads, reserve), threads) +
           eval_rest_bytes(a.ch, a.cam);
}

// k_eval_checked has no drawing queues (EvalArgs::qcap is 0 there).
size_t eval_checked_smem_bytes(const EvalArgs &a, int threads)
{
    return front_smem_bytes(a.ch.n_inst, a.qcap, threads) + eval_rest_bytes(a.ch, a.cam);
}

// CTAs of one shape that an SM holds: 1024 threads at the kernel's 64 registers,
// 228 KB of shared memory (a KB per CTA is reserved, and a little is static).
static int eval_ctas_per_sm(const ChainDev &ch, const CamDev &cam, int threads, int qcap, size_t reserve)
{
    const size_t smem = front_smem_bytes(ch.n_inst, qcap, threads) + eval_rest_bytes(ch, cam) + reserve;
    return (int)std::min<size_t>(1024 / threads, 228 * 1024 / smem);
}

// Entries per warp of the drawing queue: one per lane, or as many (16 at least)
// as leave an SM as many CTAs: at 700x493 a full queue would cost it the fourth,
// and with it a population of 64 the single wave of its clusters (51.6 us, with
// 24 entries 37.7).  8 where the image's bitmap leaves no more.
int eval_queue_cap(const ChainDev &ch, const CamDev &cam, int threads, size_t reserve)
{
    int cap = 32;
    while (cap > 16 &&
           eval_ctas_per_sm(ch, cam, threads, cap, reserve) < eval_ctas_per_sm(ch, cam, threads, 16, reserve))
        cap -= 4;
    return front_smem_bytes(ch.n_inst, cap, threads) + eval_rest_bytes(ch, cam) <= 227 * 1024 ? cap : 8;
}

// Threads per CTA that fill an SM (1024 at the kernel's 64 registers) when its
// shared memory holds few of the image's bitmaps: 256 where four fit, 512 for
// two or three, 1024 for one.  Two instruments of 40k triangles, 256 candidates,
// one CTA each: 1280x1024 742 us with 256 threads, 470 with 512, 383 with 1024;
// 960x768 410 and 350; 800x600 370 and 302 (320 threads, three to an SM: 352).
int eval_wide_threads(const ChainDev &ch, const CamDev &cam, size_t reserve)
{
    for (int n = 4; n; n /= 2)
        if (eval_ctas_per_sm(ch, cam, 1024 / n, 16, reserve) == n) return 1024 / n;
    return 256;
}

// Clusters of every size that are resident at once.
cudaError_t eval_cluster_fit(LaunchCfg &cfg)
{
    for (int k = 1; k <= cfg.cluster; ++k) {
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(k, 1, 1);
        lc.blockDim = dim3(cfg.threads, 1, 1);
        lc.dynamicSmemBytes = cfg.smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = k;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        lc.attrs = attr;
        lc.numAttrs = 1;
        const cudaError_t e = cfg.threads > 256 ? cudaOccupancyMaxActiveClusters(&cfg.fit[k], k_eval_wide, &lc)
                                                : cudaOccupancyMaxActiveClusters(&cfg.fit[k], k_eval, &lc);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// CTAs per candidate of a population of lam: as many as leave all its clusters
// resident at once.  More CTAs shorten a candidate's way but cost it barriers and
// bitmaps, so a second wave pays only with much work per thread and waves
// nearly full.  20k triangles, CTAs 1/2/4/8 (us): 640x512 64 candidates 108/62/43/41, 128
// candidates 108/70/62/69, 256 candidates 127/109/99/122; 960x768 91/56/56/83, 91/80/100/153,
// 144/145/169/282; 1280x1024 90/61/93/206, 89/115/178/375, 170/222/341/717.
static int eval_cluster(const LaunchCfg &cfg, int lam)
{
    int k = cfg.cluster;
    if (cfg.fit[1] <= 0) return k;
    while (k > 1 && lam > cfg.fit[k]) --k;
    if (cfg.threads == 256 && k <= 2 && 2 * k <= cfg.cluster && lam <= cfg.fit[k] && cfg.fit[2 * k] > 0 &&
        cfg.work >= 24LL * 2 * k * cfg.threads) {
        const int fit = cfg.fit[2 * k], waves = (lam + fit - 1) / fit;
        if (5 * lam >= 4 * waves * fit) k *= 2;
    }
    return k;
}

int eval_max_threads() { return 1024; }

cudaError_t prepare_eval(size_t smem, int threads)
{
    return ensure_smem_attr(threads > 256 ? (const void *)k_eval_wide : (const void *)k_eval, smem);
}

cudaError_t launch_eval_checked(const EvalArgs &a, const LaunchCfg &cfg, cudaStream_t s)
{
    if (a.lam == 0) return cudaSuccess;
    cudaError_t e = ensure_smem_attr((const void *)k_eval_checked, cfg.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cfg.cluster, a.lam, 1);
    lc.blockDim = dim3(cfg.threads, 1, 1);
    lc.dynamicSmemBytes = cfg.smem;
    lc.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cfg.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, k_eval_checked, a);
}

cudaError_t launch_eval(const EvalArgs &a0, const LaunchCfg &cfg, cudaStream_t s)
{
    if (a0.lam == 0) return cudaSuccess;
    if (!a0.prims) return cudaErrorInvalidValue;  // k_eval draws the primitive records (apply_mesh)
    EvalArgs a = a0;
    a.qcap = eval_queue_cap(a.ch, a.cam, cfg.threads);
    const int cluster = eval_cluster(cfg, a.lam);
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cluster, a.lam, 1);
    lc.blockDim = dim3(cfg.threads, 1, 1);
    lc.dynamicSmemBytes = cfg.smem;
    lc.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // fused generations follow each other: overlap the next one's launch with
    // this one's tail (see griddep_wait)
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = a.cma_st ? 1 : 0;
    lc.attrs = attr;
    lc.numAttrs = 2;
    return cfg.threads > 256 ? cudaLaunchKernelEx(&lc, k_eval_wide, a) : cudaLaunchKernelEx(&lc, k_eval, a);
}

// ----------------------------------------------------------------------------
// Mask packing: one warp per 32-pixel word, coverage by __ballot_sync.
// ----------------------------------------------------------------------------
__global__ void k_pack_mask(const uint8_t *mask, uint32_t *packed, int W, int H, int Wq)
{
    long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (gw >= (long long)H * Wq) return;
    int i = (int)(gw / Wq), w = (int)(gw - (long long)i * Wq);
    int j = w * 32 + lane;
    bool on = (j < W) && mask[(size_t)i * W + j] != 0;
    unsigned b = __ballot_sync(0xffffffffu, on);
    if (lane == 0) packed[gw] = b;
}

cudaError_t launch_pack_mask(const uint8_t *mask, uint32_t *packed, int W, int H, int Wq, cudaStream_t s)
{
    long long threads = (long long)H * Wq * 32;
    int blocks = (int)((threads + 255) / 256);
    if (blocks == 0) return cudaSuccess;
    k_pack_mask<<<blocks, 256, 0, s>>>(mask, packed, W, H, Wq);
    return cudaGetLastError();
}

}  // namespace trk
