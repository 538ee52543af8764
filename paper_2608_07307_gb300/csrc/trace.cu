// trace.cu -- ray generation, first-hit traversal, SRP shading, specular
// bounces and the force / torque reduction (Sec. 4.3, 6.1).
//
// k_frame.  Once per slot: the window (u, v bounds from the vertex pass), the
// FP32 ray generation, the error bounds of the FP32 decisions and the
// per-part traversal views, into a small context every trace block copies;
// in launches of few slots its extra blocks also clear the pixel keys
// (k_clear_keys otherwise).
//
// k_raster / k_raster_big / k_raster_chunks / k_raster_pass1 (primary visibility).  All primary
// rays of an evaluation are parallel, so each triangle applies the trace's own
// FP32 view-frame test (prim_test) to the pixel centres inside its projected
// box: pass 0 keeps the nearest certain hit per pixel (64-bit atomic minimum of
// depth bits and triangle), pass 1 lists the triangles whose decision there was
// uncertain against it.  Large projected triangles are rasterised in 16 x 16
// pixel chunks, a warp each, listing only the chunks that can meet them
// (k_raster_pass1: the second pass over both kinds in one launch).
//
// k_trace (FP32 fast path).  A block is four warps, each over a 32-pixel tile
// (8 x 4 by default; the shape is chosen per mesh, grid and bounce count by the
// autotuner), sharing one copy of the slot context.  The tiles of every slot of
// a launch form one flat grid, so one launch can trace different meshes, grid
// sizes and bounce counts.  The primary segment takes the raster's nearest
// certain hit and candidates (a pixel with too many candidates, those past two where
// the slot's list of them ran over, or every pixel when rasterisation is off, traverses
// instead).  Every traversed segment walks
// each part's 4-wide BVH (128 B nodes: six float4 of child boxes in SoA order,
// the near and far planes picked by the ray's octant, and the child refs),
// parts in the order the ray enters their root boxes, with the watertight
// ray/triangle test (Woop, Benthin and Wald, "Watertight ray/triangle
// intersection", JCGT 2(1), 2013):
//   * primary rays share the direction d, so their test runs in the view frame
//     (u, v, d): per-vertex projections computed in FP64 and rounded once to
//     FP32, the ray is the line through the pixel centre (uc, vc) along the
//     third axis, and the watertight shear vanishes;
//   * secondary (specular) rays use the world-frame test with the shear; their
//     origin is rebuilt from the hit's barycentric weights, and they pass over
//     the subtree of their origin's coplanar group.
// Every FP32 decision carries an error bound: when an edge function, the
// nearest-hit comparison or the self-hit threshold is within its bound, the
// triangle is settled in FP64 at the end of the segment (resolve64); only a ray
// with too many such triangles, or that hits one without an FP32 normal, is handed
// to the FP64 re-trace and contributes nothing here.  Per hit:
// absorbed + specular + Lambertian momentum, torque about c_ref, specular ray
// of weight w rho_s.  Per-ray sums in FP32 (at most 1 + bounces terms), tile
// sums by an FP32 butterfly and integer reductions, one partial per tile; the
// tile's handed-off rays go to its own list slot.
//
// resolve64 (FP64, inside k_trace).  When a segment had FP32 decisions within
// their bounds, its uncertain triangles and its nearest certain hit are tested
// again in FP64 against the exact ray of the segment (rare: ~0.5% of the rays
// of a 200k-triangle mesh at 1024^2).
//
// k_trace_few (launches of few slots).  The same trace with a block per tile: the
// block's first warp settles and shades, and the rays that go on are walked by
// its warps, eight to sixteen rays a warp with all lanes (walk_warp): the open
// (ray, node) pairs are shared out a lane a pair, so a long walk does not hold
// up its warp.  Same decisions, same bits.
//
// FP64 re-trace (in k_reduce1).  A ray whose uncertain triangles overflow the
// candidate list, or whose hit has no FP32 normal, is re-traced from its pixel definition with FP64 rays and
// vertices, the same BVH (boxes padded well beyond the FP32 rounding of the
// ray; leaves pre-tested in FP32 with a bound, so only triangles not certainly
// missed are tested in FP64) and the same watertight test in FP64.
//
// k_reduce1 (+ k_reduce after diffuse rays).  Fixed-order FP64 sums: contiguous
// ranges of tile partials (and the re-traced rays of those tiles) per
// first-level block, then those per evaluation in block order, by the last
// first-level block of the evaluation to finish (an atomic ticket; without
// diffuse rays) or by k_reduce, scaled by P0 / dist^2 times the pixel area.  No
// atomics on data: results are bit-reproducible.
//
// k_demit, k_dscan, k_diffuse (optional, Sec. 6.1's diffuse rays).  After the re-trace,
// a thread per primary ray replays its specular chain in FP64 through the recorded hit
// triangles and writes a record per hit that emits; the records are counted; then a
// thread per (record, sample) traces its sample of the K cosine-weighted diffuse rays
// (SplitMix64 stream) in FP32 with the same error bounds (walk_warp: incoherent rays,
// whose lanes would wait for each other), settling the uncertain triangles in FP64
// (settle64); its per-block FP64 sums are added by k_reduce in a fixed order.
//
// k_bvh_check (diagnostics).  One thread per part walks slot 0's 4-wide tree and counts
// leaf references, child boxes outside their parent's and triangles outside their leaf.
#include <math.h>
#include <stddef.h>

#include <algorithm>

#include "srp_internal.cuh"

namespace srp {

constexpr float kU = 5.9604645e-8f;  // unit roundoff of FP32, 2^-24
constexpr int kWalkRefBits = 27;      // of a walk entry, for the part and its node or triangle (walk_warp)
constexpr int kWalkDepth = 30;        // levels a walk's order keys hold
// k_trace_few: warps a block (a tile), resident blocks.  50k / 200k triangles, 512^2, 1 bounce, us: 2 warps at 8
// blocks 75 / 87, 10 blocks 79 / 92, 12 blocks 83 / 99 (spills); 4 warps at 6 blocks 81 / 91, 1 warp at 20 125 / 153.
constexpr int kFewWarps = 2, kFewBlocksPerSM = 8;

struct PartView {
    const float4 *node;
    const float4 *tri;   // world-frame triangle records
    const int4 *v4;      // vertex ids of the part's sorted triangles
    const double *v64;   // v64[3 * (vi - vert_begin) + c]
    int root;            // 0, or ~0 for a one-triangle part
    int limit;           // bound on loop iterations of one part walk (nodes + triangles)
    int tri_begin, vert_begin;
    float box[6];        // root box (filled when a block loads the context, from box_src)
    const float *box_src;  // the part's root box: the refit's output for a dynamic part with triangles
};

struct TraceCtx {
    // FP32 ray generation: o = org + (i+.5) du + (j+.5) dv; view-frame pixel centres
    float org[3], du[3], dv[3], dir[3];
    float umin32, vmin32, du32, dv32, w0_32;
    float rdu32, rdv32;    // 1 / du32, 1 / dv32 (the raster's conservative pixel boxes)
    float delta_p, tau_p;  // primary: bound on view-frame coordinate error, band on t
    float delta_s;         // secondary: origin-error term added per segment
    float R, L, pad, eps32;
    float cref32[3];
    int n_parts, n_mats;
    int ref_bits;          // bits of a node or triangle in a walk entry (walk_warp); 0: a part has too many
    int walk_bound;        // bound on the batches of a walk
    int walk_spare;        // node list entries kept for a depth-first walk at the end of the room
    int skip;              // evaluation skipped (kSkip...): trace blocks only clear their hand-off count
    const float4 *vview;   // slot's view-frame vertices
    const double *vview64; // the same in FP64
    const float2 *mat32;
    const double *mat64;
    const unsigned *tri_mat;
    const int *tri_vidx;
    const int2 *grp;  // per sorted triangle: subtree of its coplanar group, deviation bound
    const int4 *tri_v4;    // vertex ids of the sorted triangles (the raster's first load)
    int n_tris;
    // FP64 window and basis for the FP64 path
    double umin, vmin, wmin, Du, Dv, Lw, eps;
    double rN;  // 1 / N when N is a power of two (dividing by N is then exactly this product), else 0
    double u[3], v[3], d[3], c_ref[3];
    PartView part[kMaxParts];
};

size_t trace_ctx_bytes() { return sizeof(TraceCtx); }

// The trace kernels' dynamic shared memory: the slot context up to the most
// parts of the launch's slots (16-byte rounded), then the per-thread hit
// columns of the most segments; sized per launch so that the blocks an SM runs
// fit the small shared-memory configuration the kernels ask for.
__host__ __device__ __forceinline__ int trace_parts_cap(int ctx_parts)
{
    return ctx_parts > 0 && ctx_parts < kMaxParts ? ctx_parts : kMaxParts;
}
__host__ __device__ __forceinline__ size_t trace_ctx_dyn_bytes(int ctx_parts)
{
    return (offsetof(TraceCtx, part) + (size_t)trace_parts_cap(ctx_parts) * sizeof(PartView) + 15) / 16 * 16;
}
__host__ __device__ __forceinline__ size_t trace_dyn_bytes(int ctx_parts, int hpt_segs)
{
    const int ns = hpt_segs > 0 && hpt_segs < kMaxBounces + 1 ? hpt_segs : kMaxBounces + 1;
    return trace_ctx_dyn_bytes(ctx_parts) + (size_t)ns * 128 * sizeof(int);
}

// x / N, as a product when N is a power of two (the same value, without an FP64 division)
__device__ __forceinline__ double pix64(double x, double rN, int N) { return rN != 0.0 ? x * rN : x / N; }

__device__ __forceinline__ float pick(float x, float y, float z, int k) { return k == 0 ? x : (k == 1 ? y : z); }
__device__ __forceinline__ double pickd(double x, double y, double z, int k) { return k == 0 ? x : (k == 1 ? y : z); }

// ------------------------------------------------------------- k_frame
__global__ void k_frame(TraceArgs a)
{
    pdl_enter();
    // every load first, then the arithmetic and the stores: a load placed after
    // a store it might alias waits for everything before it, and a chain of such
    // round trips, not the arithmetic, would set this kernel's duration
    const int s = blockIdx.x, lane = threadIdx.x;
    // launches of few slots: every block of the slot sets the pixel keys to all
    // ones (no hit, no candidate) for the raster
    if (a.raster && a.pix_key) {
        unsigned long long *key = a.pix_key + (size_t)s * a.ray_stride;
        const size_t stride = (size_t)gridDim.y * blockDim.x;
        for (size_t i = (size_t)blockIdx.y * blockDim.x + threadIdx.x; i < a.ray_stride; i += stride) key[i] = ~0ull;
    }
    if (blockIdx.y != 0 || lane >= 32) return;  // the context: one warp of the slot
    const SlotDesc &D = a.sd[s];
    const MeshDev *m = D.mesh;
    const SlotBufs sb = D.sb;
    const int N = D.N;
    const SlotPose &P = a.pose[s];
    const int skip = P.skip;
    const int np = m->n_parts;
    PartInfo pi{};
    if (lane < kMaxParts) pi = m->part[lane];
    // walk entries: the ray in five bits, the part in as few as the parts need, the rest for the node or triangle
    const int ref_bits = kWalkRefBits - (32 - __clz(np - 1));
    const int stack_need = m->stack_need;
    const bool refs_fit = __all_sync(0xffffffffu, lane >= np || pi.tri_count <= (1 << ref_bits));
    const float *box_static = lane < kMaxParts ? m->root_box_static[lane] : nullptr;
    const int4 *tri_v4 = m->tri_v4;
    const int n_tris = m->n_tris;
    const float4 *node_static = m->node_static, *tri_static = m->tri_static;
    const double *rest64 = m->rest64;
    // a component a lane (of three): an FP64 instruction costs the warp the same for one lane or all
    const int c3 = lane % 3;
    const double lo = ord_to_dbl(P.wmin_bits[c3]), hi = ord_to_dbl(P.wmax_bits[c3]);
    const double u3 = P.u[c3], v3 = P.v[c3], d3 = P.d[c3], cref = m->c_ref[c3];
    double Rm = 0.0, pad = 0.0;
    int n_mats = 0;
    const float2 *mat32 = nullptr;
    const double *mat64 = nullptr;
    const unsigned *tri_mat = nullptr;
    const int *tri_vidx = nullptr;
    const int2 *grp = nullptr;
    if (lane == 0) {
        Rm = m->R;
        pad = m->pad;
        n_mats = m->n_mats;
        mat32 = m->mat32;
        mat64 = m->mat64;
        tri_mat = m->tri_mat;
        tri_vidx = m->tri_vidx;
        grp = m->grp;
    }
    TraceCtx &B = reinterpret_cast<TraceCtx *>(a.tctx)[s];
    if (lane == 0) {
        B.skip = skip;
        if (a.raster) {
            a.rast_bad[s] = 0;
            a.pix_over[(size_t)s * kOverWords] = 0u;
            if (s == 0) { *a.big_count = 0u; *a.bigt_count = 0u; }
        }
        if (a.queue) {
            for (int k = 0; k < 3; k++) a.qstate[kQSlot + 3 * s + k] = 0u;
            if (s == 0) { a.qstate[kQHead] = 0u; a.qstate[kQAbort] = 0u; }
        }
        B.n_parts = np;
        B.ref_bits = refs_fit && stack_need <= 3 * kWalkDepth + 1 ? ref_bits : 0;
        B.walk_spare = stack_need;
        B.walk_bound = a.walk_limit_test ? 1 : (int)min(64ll * n_tris + 4096ll, 0x7fffffffll);
        if (a.red_ticket) a.red_ticket[s] = 0u;
    }
    // the parts' traversal views, a lane each (in a skipped slot too: its context is copied by blocks that find out
    // then, and the copy follows box_src)
    if (lane < np) {
        PartView &pv = B.part[lane];
        pv.root = pi.tri_count > 1 ? 0 : ~0;
        pv.limit = a.walk_limit_test ? 1 : pi.node_count + pi.tri_count + 8;
        pv.tri_begin = pi.tri_begin;
        pv.vert_begin = pi.vert_begin;
        pv.v4 = tri_v4 + pi.tri_begin;
        if (pi.dynamic && pi.tri_count > 0) {
            pv.node = sb.node + (size_t)pi.dyn_node_off * kNode4;
            pv.tri = sb.tri + (size_t)pi.dyn_tri_off * 3;
            pv.v64 = sb.vert64 + (size_t)pi.dyn_vert_off * 3;
            pv.box_src = sb.root_box + (size_t)lane * 6;
        } else {
            pv.node = node_static + (size_t)pi.node_begin * kNode4;
            pv.tri = tri_static + (size_t)pi.tri_begin * 3;
            pv.v64 = rest64 + (size_t)pi.vert_begin * 3;
            pv.box_src = box_static;
        }
    }
    if (skip) return;
    const auto all = [](double x, int l) { return __shfl_sync(0xffffffffu, x, l); };
    const double umin = all(lo, 0), umax = all(hi, 0), vmin = all(lo, 1), vmax = all(hi, 1), wmin = all(lo, 2),
                 wmax = all(hi, 2);
    const double D3 = hi - lo;
    const double Du = all(D3, 0), Dv = all(D3, 1), Dw = all(D3, 2);
    const double Lw = sqrt(Du * Du + Dv * Dv + Dw * Dw);
    const double eps = a.eps_rel * Lw;
    const double qn = (lane == 0 ? Du : lane == 1 ? Dv : 1.0) / N;  // the pixel's sides and 1 / N
    const double DuN = all(qn, 0), DvN = all(qn, 1), rN = all(qn, 2);
    const double w0 = wmin - kStandoff;
    const double o3 = umin * u3 + vmin * v3 + w0 * d3;
    if (lane < 3) {
        B.org[lane] = (float)o3;
        B.du[lane] = (float)(DuN * u3);
        B.dv[lane] = (float)(DvN * v3);
        B.dir[lane] = (float)d3;
        B.u[lane] = u3; B.v[lane] = v3; B.d[lane] = d3;
        B.c_ref[lane] = cref;
        B.cref32[lane] = (float)cref;
    }
    if (lane != 0) return;
    B.umin = umin; B.vmin = vmin; B.wmin = wmin;
    B.rN = (N & (N - 1)) == 0 ? rN : 0.0;
    B.Du = Du; B.Dv = Dv;
    B.Lw = Lw;
    B.eps = eps;
    B.eps32 = (float)eps;
    B.umin32 = (float)umin; B.vmin32 = (float)vmin;
    B.du32 = (float)DuN; B.dv32 = (float)DvN;
    B.rdu32 = 1.0f / B.du32; B.rdv32 = 1.0f / B.dv32;
    B.w0_32 = (float)w0;
    const double u = 5.9604644775390625e-8;
    // Primary (view frame): vertex projections rounded once (|p| u/2), pixel
    // centres from rounded umin, du and one FMA, differences rounded; the bound
    // doubles that sum.
    const double Mw = fmax(fmax(fabs(umin), fabs(umax)), fmax(fabs(vmin), fabs(vmax)));
    const double Dm = fmax(Du, Dv);
    const float delta_p = (float)(2.0 * u * (3.0 * Mw + 2.0 * Dm));
    B.delta_p = delta_p;
    const double Wm = fmax(fabs(wmin), fabs(wmax)) + kStandoff;
    B.tau_p = (float)(16.0 * u * Wm + 32.0 * delta_p);
    // Secondary (world frame): the origin is rebuilt from the hit's barycentric
    // weights (error ~2 x the previous bound + rounding at |x| <= R, plus the
    // rounding of posed vertices); the per-triangle terms (subtraction, shear,
    // reflected direction) are added in the test from that triangle's distance.
    B.delta_s = (float)(6.0 * u * Rm);
    B.R = (float)Rm;
    B.L = (float)Lw;
    B.pad = (float)pad;
    B.n_mats = n_mats;
    B.vview = sb.vview;
    B.vview64 = sb.vview64;
    B.mat32 = mat32;
    B.mat64 = mat64;
    B.tri_mat = tri_mat;
    B.tri_vidx = tri_vidx;
    B.grp = grp;
    B.tri_v4 = tri_v4;
    B.n_tris = n_tris;
}

// Copy the slot context (header + the parts in use) into shared memory.
__device__ __forceinline__ void load_ctx(TraceCtx &B, const TraceArgs &a, int s)
{
    const TraceCtx *g = reinterpret_cast<const TraceCtx *>(a.tctx) + s;
    // the record up to its last used part view (the part count from the record itself)
    const int np = __ldg(&g->n_parts);
    const int words = (int)((offsetof(TraceCtx, part) + np * sizeof(PartView)) / 4);
    const int *src = reinterpret_cast<const int *>(g);
    int *dst = reinterpret_cast<int *>(&B);
    for (int k = threadIdx.x; k < words; k += blockDim.x) dst[k] = __ldg(src + k);
    __syncthreads();
    // the root boxes, from where the refit (or the mesh load) left them: the
    // frame kernel that wrote the context did not wait for the refit
    for (int k = threadIdx.x; k < 6 * np; k += blockDim.x) B.part[k / 6].box[k % 6] = B.part[k / 6].box_src[k % 6];
}

// Slab test of one box; returns entry t or +inf.
__device__ __forceinline__ float box_enter(float lx, float hx, float ly, float hy, float lz, float hz, const float *inv,
                                           const float *oi, float tlo, float thi)
{
    float x0 = fmaf(lx, inv[0], -oi[0]), x1 = fmaf(hx, inv[0], -oi[0]);
    float y0 = fmaf(ly, inv[1], -oi[1]), y1 = fmaf(hy, inv[1], -oi[1]);
    float z0 = fmaf(lz, inv[2], -oi[2]), z1 = fmaf(hz, inv[2], -oi[2]);
    float tn = fmaxf(fmaxf(fminf(x0, x1), fminf(y0, y1)), fmaxf(fminf(z0, z1), tlo));
    float tf = fminf(fminf(fmaxf(x0, x1), fmaxf(y0, y1)), fminf(fmaxf(z0, z1), thi));
    return tn <= tf ? tn : INFINITY;
}

// Slab test of one box given its near and far plane on each axis (the planes
// the ray meets first and last): no per-axis ordering needed.
__device__ __forceinline__ float box_enter_nf(float nx, float fx, float ny, float fy, float nz, float fz,
                                              const float *inv, const float *oi, float tlo, float thi)
{
    float tn = fmaxf(fmaxf(fmaf(nx, inv[0], -oi[0]), fmaf(ny, inv[1], -oi[1])), fmaxf(fmaf(nz, inv[2], -oi[2]), tlo));
    float tf = fminf(fminf(fmaf(fx, inv[0], -oi[0]), fmaf(fy, inv[1], -oi[1])), fminf(fmaf(fz, inv[2], -oi[2]), thi));
    return tn <= tf ? tn : INFINITY;
}

__device__ __forceinline__ void cswap(float &ta, int &ra, float &tb, int &rb)
{
    if (tb < ta) {
        float t = ta; ta = tb; tb = t;
        int r = ra; ra = rb; rb = r;
    }
}

// One 4-wide node: slab tests of its four child boxes (lo.x, hi.x, lo.y, hi.y,
// lo.z, hi.z in float4 0..5, one lane per child; child refs in float4 6).
// Bit k of oct is 1 where the ray runs backwards along axis k: the near plane is then
// the box's upper bound, so picking the float4 by address replaces the per-axis
// min/max of the slab test.  An unused slot's box (+inf, -inf) is entered at
// +inf and never hit.  Continues with the nearest child entered and pushes the
// others, farthest first.  Returns the number of children entered (0: pop the
// stack), -1 when the stack would overflow.
__device__ __forceinline__ int node4_step(const float4 *nd, const float *inv, const float *oi, int oct,
                                          float tlo, float thi, int &ref, int *stack, int &sp)
{
    const int ox = oct & 1, oy = (oct >> 1) & 1, oz = (oct >> 2) & 1;
    float4 nx = __ldg(nd + ox), fx = __ldg(nd + 1 - ox), ny = __ldg(nd + 2 + oy),
           fy = __ldg(nd + 3 - oy), nz = __ldg(nd + 4 + oz), fz = __ldg(nd + 5 - oz);
    int4 c = __ldg(reinterpret_cast<const int4 *>(nd + 6));
    float ta = box_enter_nf(nx.x, fx.x, ny.x, fy.x, nz.x, fz.x, inv, oi, tlo, thi);
    float tb = box_enter_nf(nx.y, fx.y, ny.y, fy.y, nz.y, fz.y, inv, oi, tlo, thi);
    float tc = box_enter_nf(nx.z, fx.z, ny.z, fy.z, nz.z, fz.z, inv, oi, tlo, thi);
    float td = box_enter_nf(nx.w, fx.w, ny.w, fy.w, nz.w, fz.w, inv, oi, tlo, thi);
    int ra = c.x, rb = c.y, rc = c.z, rd = c.w;
    cswap(ta, ra, tb, rb);
    cswap(tc, rc, td, rd);
    cswap(ta, ra, tc, rc);
    cswap(tb, rb, td, rd);
    cswap(tb, rb, tc, rc);
    if (ta == INFINITY) return 0;
    const int n = 1 + (tb != INFINITY) + (tc != INFINITY) + (td != INFINITY);
    if (sp + n - 1 > kStack) return -1;
    if (td != INFINITY) stack[sp++] = rd;
    if (tc != INFINITY) stack[sp++] = rc;
    if (tb != INFINITY) stack[sp++] = rb;
    ref = ra;
    return n;
}

struct Ray32 {
    float o[3], d[3], inv[3], oi[3];
    float Sx, Sy, Sz;
    // bits 0-2: 1 where the direction component is negative (the ray's octant);
    // bits 3-4, 5-6, 7-8: the axes kx, ky, kz of the watertight test (one
    // register instead of six)
    int code;
    __device__ __forceinline__ int kx() const { return (code >> 3) & 3; }
    __device__ __forceinline__ int ky() const { return (code >> 5) & 3; }
    __device__ __forceinline__ int kz() const { return (code >> 7) & 3; }
};

__device__ __forceinline__ void ray_setup(Ray32 &r)
{
    int oct = 0;
    for (int k = 0; k < 3; k++) {
        float dk = r.d[k];
        float ds = fabsf(dk) < 1e-20f ? copysignf(1e-20f, dk) : dk;
        r.inv[k] = 1.0f / ds;
        r.oi[k] = r.o[k] * r.inv[k];
        oct |= (r.inv[k] < 0.f ? 1 : 0) << k;
    }
    float ax = fabsf(r.d[0]), ay = fabsf(r.d[1]), az = fabsf(r.d[2]);
    int kz = (ax > ay) ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    int kx = kz == 2 ? 0 : kz + 1;
    int ky = kx == 2 ? 0 : kx + 1;
    float dz = pick(r.d[0], r.d[1], r.d[2], kz);
    if (dz < 0.f) { int t = kx; kx = ky; ky = t; }
    r.code = oct | (kx << 3) | (ky << 5) | (kz << 7);
    r.Sx = pick(r.d[0], r.d[1], r.d[2], kx) / dz;
    r.Sy = pick(r.d[0], r.d[1], r.d[2], ky) / dz;
    r.Sz = 1.0f / dz;
}

// FP32 view-frame test of one triangle against the primary ray through pixel
// centre (uc, vc): the ray is the third axis, so the edge functions are 2-D
// cross products of the projected vertices (u, v, depth in a, b, c) relative
// to the centre.  Error bounds from the coordinate error delta of the rounded
// projections and centre, plus the rounding of the products.
struct Prim32 {
    float U, V, W, eU, eV, eW, det, T;
};

// The edge functions, determinant and scaled depth without the bounds.
__device__ __forceinline__ Prim32 prim_core(float4 a, float4 b, float4 c, float uc, float vc, float w0)
{
    Prim32 q;
    float Ax = a.x - uc, Ay = a.y - vc, Bx = b.x - uc, By = b.y - vc, Cx = c.x - uc, Cy = c.y - vc;
    q.U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    q.V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    q.W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    q.eU = q.eV = q.eW = 0.0f;
    q.det = q.U + q.V + q.W;
    q.T = fmaf(q.U, a.z - w0, fmaf(q.V, b.z - w0, q.W * (c.z - w0)));
    return q;
}

__device__ __forceinline__ Prim32 prim_test(float4 a, float4 b, float4 c, float uc, float vc, float delta, float w0)
{
    const float u4 = 4.0f * kU;
    Prim32 q;
    float Ax = a.x - uc, Ay = a.y - vc, Bx = b.x - uc, By = b.y - vc, Cx = c.x - uc, Cy = c.y - vc;
    q.U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    q.V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    q.W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    q.eU = delta * (fabsf(Bx) + fabsf(By) + fabsf(Cx) + fabsf(Cy)) + u4 * (fabsf(Cx * By) + fabsf(Cy * Bx));
    q.eV = delta * (fabsf(Ax) + fabsf(Ay) + fabsf(Cx) + fabsf(Cy)) + u4 * (fabsf(Ax * Cy) + fabsf(Ay * Cx));
    q.eW = delta * (fabsf(Ax) + fabsf(Ay) + fabsf(Bx) + fabsf(By)) + u4 * (fabsf(Bx * Ay) + fabsf(By * Ax));
    q.det = q.U + q.V + q.W;
    q.T = fmaf(q.U, a.z - w0, fmaf(q.V, b.z - w0, q.W * (c.z - w0)));
    return q;
}

struct Best32 {
    float t;
    int part, tl;
    float b1, b2;  // barycentric weights of the hit's second and third vertex
};

struct Counts {
    unsigned nodes, tris, boxes;
    unsigned why[4];  // uncertain FP32 decisions: primary edge, secondary edge, near tie, self-hit band
    int flags;
};

// Triangles whose FP32 decision was not certain, for the FP64 resolution at the
// end of the segment (part << 24 | part-local triangle).  The list lives in
// shared memory, one column per lane (entry c at id[c * kCandStride]) of a
// warp-wide array: a per-thread array indexed at run time would sit in local
// memory, and its traffic would compete with the node fetches in L1.
constexpr int kCand = 8;
constexpr int kLaneStride = 128;  // threads of the kernels that keep per-thread columns in shared memory
struct Cands {
    int n;
    int *id;
};
constexpr int kCandStride = 32;  // lanes' candidate columns: a warp's lists side by side

__device__ __forceinline__ bool push_cand(Cands &c, int p, int tl)
{
    if (c.n >= kCand) return false;
    c.id[c.n * kCandStride] = (p << 24) | tl;
    c.n++;
    return true;
}

// Classify one candidate from its edge functions and depth.  Certain misses and
// certain hits are settled here (best keeps the nearest certain hit); a triangle
// whose decision is within its bound becomes a candidate of the FP64 resolution,
// and so does the best hit it displaces within the tie band.  Returns false when
// the candidate list overflows (the ray then goes to the FP64 re-trace).
template <bool COUNT>
__device__ __forceinline__ bool classify(float U, float V, float W, float eU, float eV, float eW, float T, float det,
                                         float tlo, float tau, int p, int tl, Best32 &best, bool primary, Counts &cn,
                                         Cands &cd)
{
    bool neg = (U < -eU) || (V < -eV) || (W < -eW);
    bool pos = (U > eU) || (V > eV) || (W > eW);
    if (neg && pos) return true;  // certainly outside
    bool unsure = fabsf(U) <= eU || fabsf(V) <= eV || fabsf(W) <= eW;
    float t = T / det;
    if (unsure) {
        // near an edge: matters unless the plane is certainly behind the origin or beyond the best hit
        bool far = (fabsf(det) > 1e-30f) && (t > best.t + tau || t < tlo - tau);
        if (far) return true;
        if (COUNT) cn.why[primary ? 0 : 1]++;
        return push_cand(cd, p, tl);
    }
    bool amb = false;
    if (fabsf(t - tlo) <= tau) { amb = true; if (COUNT) cn.why[3]++; }
    else if (fabsf(t - best.t) <= tau) { amb = true; if (COUNT) cn.why[2]++; }
    if (amb && !push_cand(cd, p, tl)) return false;
    if (t > tlo && t < best.t) {
        if (amb && best.part >= 0 && !push_cand(cd, best.part, best.tl)) return false;
        float id = 1.0f / det;
        best.t = t; best.part = p; best.tl = tl; best.b1 = V * id; best.b2 = W * id;
    }
    return true;
}

// World-frame watertight test of a secondary ray against one triangle record:
// the vertices sheared onto the ray's axes, the edge functions, and the bound
// on the coordinate error (origin error delta + subtraction, shear and
// reflected-direction rounding, growing with this triangle's distance).
struct Shear32 {
    float Ax, Ay, Bx, By, Cx, Cy, Akz, Bkz, Ckz, U, V, W;
    float dc, Mv;  // the bound; the largest sheared coordinate
};
struct ShearRay {
    float o[3], Sx, Sy, Sz;
    int code;  // as Ray32
    __device__ __forceinline__ int kx() const { return (code >> 3) & 3; }
    __device__ __forceinline__ int ky() const { return (code >> 5) & 3; }
    __device__ __forceinline__ int kz() const { return (code >> 7) & 3; }
};
template <class R>
__device__ __forceinline__ Shear32 shear_test(const R &r, float4 a, float4 b, float4 c, float delta)
{
    Shear32 q;
    float A0 = a.x - r.o[0], A1 = a.y - r.o[1], A2 = a.z - r.o[2];
    float B0 = b.x - r.o[0], B1 = b.y - r.o[1], B2 = b.z - r.o[2];
    float C0 = c.x - r.o[0], C1 = c.y - r.o[1], C2 = c.z - r.o[2];
    q.Akz = pick(A0, A1, A2, r.kz()); q.Bkz = pick(B0, B1, B2, r.kz()); q.Ckz = pick(C0, C1, C2, r.kz());
    q.Ax = fmaf(-r.Sx, q.Akz, pick(A0, A1, A2, r.kx())); q.Ay = fmaf(-r.Sy, q.Akz, pick(A0, A1, A2, r.ky()));
    q.Bx = fmaf(-r.Sx, q.Bkz, pick(B0, B1, B2, r.kx())); q.By = fmaf(-r.Sy, q.Bkz, pick(B0, B1, B2, r.ky()));
    q.Cx = fmaf(-r.Sx, q.Ckz, pick(C0, C1, C2, r.kx())); q.Cy = fmaf(-r.Sy, q.Ckz, pick(C0, C1, C2, r.ky()));
    q.U = __fsub_rn(__fmul_rn(q.Cx, q.By), __fmul_rn(q.Cy, q.Bx));
    q.V = __fsub_rn(__fmul_rn(q.Ax, q.Cy), __fmul_rn(q.Ay, q.Cx));
    q.W = __fsub_rn(__fmul_rn(q.Bx, q.Ay), __fmul_rn(q.By, q.Ax));
    const float mxy = fmaxf(fmaxf(fabsf(q.Ax), fabsf(q.Bx)), fabsf(q.Cx)),
                myy = fmaxf(fmaxf(fabsf(q.Ay), fabsf(q.By)), fabsf(q.Cy));
    float dz = fmaxf(fmaxf(fabsf(q.Akz), fabsf(q.Bkz)), fabsf(q.Ckz)) + mxy + myy;
    q.dc = fmaf(16.0f * kU, dz, delta);
    q.Mv = fmaxf(mxy, myy);
    return q;
}

// A certain miss by one common bound: with M the largest |x|, |y| of the three
// vertices, every edge function's bound is at most 4 M dc + 2 M^2 u4 (the
// factor covers this sum's own rounding); an edge function beyond it on each
// side is a certain miss, as classify would find with the exact bounds.
__device__ __forceinline__ bool certain_miss(const Shear32 &q)
{
    const float u4 = 4.0f * kU;
    const float Eb = fmaf(q.dc, 4.0f * q.Mv, (2.0f * u4) * q.Mv * q.Mv) * 1.001f;
    return q.Mv > 1e-18f && fminf(fminf(q.U, q.V), q.W) < -Eb && fmaxf(fmaxf(q.U, q.V), q.W) > Eb;
}

// The exact bounds of the three edge functions.
__device__ __forceinline__ void shear_bounds(const Shear32 &q, float &eU, float &eV, float &eW)
{
    const float u4 = 4.0f * kU;
    eU = q.dc * (fabsf(q.Bx) + fabsf(q.By) + fabsf(q.Cx) + fabsf(q.Cy)) + u4 * (fabsf(q.Cx * q.By) + fabsf(q.Cy * q.Bx));
    eV = q.dc * (fabsf(q.Ax) + fabsf(q.Ay) + fabsf(q.Cx) + fabsf(q.Cy)) + u4 * (fabsf(q.Ax * q.Cy) + fabsf(q.Ay * q.Cx));
    eW = q.dc * (fabsf(q.Ax) + fabsf(q.Ay) + fabsf(q.Bx) + fabsf(q.By)) + u4 * (fabsf(q.Bx * q.Ay) + fabsf(q.By * q.Ax));
}

// Nearest hit of one segment in FP32 by one lane: the walk whose decisions
// walk_warp reproduces, run for a primary segment that the raster did not
// settle and for a secondary one that outgrows walk_warp's lists.  PRIMARY:
// the view-frame test at pixel centre (uc, vc); otherwise the world-frame test.  Triangles whose decision
// was within its error bound are collected in cd (settled in FP64 afterwards);
// returns false when they overflow the list or a walk bound is reached (the ray
// then goes to the FP64 re-trace).  A secondary ray leaving the plane of its
// origin's coplanar group passes the group's subtree (ref gskip of part gpart)
// by: none of its triangles can be hit beyond the origin.  COPY: B is a block's
// copy of the context, which has the parts' root boxes in it.
template <bool COUNT, bool PRIMARY, bool COPY>
__device__ __forceinline__ bool nearest32(const TraceCtx &B, const Ray32 &r, float uc, float vc, float tlo, int skip,
                                          int gpart, int gskip, float delta, float tau, Best32 &best, Counts &cn,
                                          Cands &cd)
{
    best.t = INFINITY;
    best.part = -1;
    best.tl = -1;
    cd.n = 0;
    int stack[kStack];
    unsigned n_nodes = 0, n_tris = 0, n_boxes = 0;
    bool clean = true;
    const float u4 = 4.0f * kU;
    // parts in the order the ray enters their root boxes: a near hit then culls
    // the parts behind it at their root
    float te[kMaxParts];
    int po[kMaxParts], np = 0;
    for (int p = 0; p < B.n_parts; p++) {
        const PartView &pv = B.part[p];
        if (p == gpart && pv.root == gskip) continue;  // the whole part is the origin's plane
        const float *box = COPY ? pv.box : pv.box_src;
        float t = box_enter(box[0], box[3], box[1], box[4], box[2], box[5], r.inv, r.oi, tlo - tau, INFINITY);
        if (t == INFINITY) continue;
        int k = np++;
        while (k > 0 && te[k - 1] > t) { te[k] = te[k - 1]; po[k] = po[k - 1]; k--; }
        te[k] = t;
        po[k] = p;
    }
    for (int q = 0; q < np; q++) {
        if (te[q] > best.t + tau) break;  // this part and every later one start beyond the best hit
        const int p = po[q];
        const PartView &pv = B.part[p];
        const int gs = p == gpart ? gskip : kNoGroup;
        int sp = 0, iters = 0;
        int ref = pv.root;
        while (true) {
            if (++iters > pv.limit) { clean = false; cn.flags |= kFlagStack; break; }
            if (ref >= 0) {
                if (ref != gs) {
                    const int n = node4_step(pv.node + (size_t)ref * kNode4, r.inv, r.oi, r.code, tlo - tau,
                                             best.t + tau, ref, stack, sp);
                    if (COUNT) { n_nodes++; n_boxes += 4; }
                    if (n < 0) { clean = false; cn.flags |= kFlagStack; break; }
                    if (n > 0) continue;
                }
            } else {
                int tl = ~ref;
                if (COUNT) n_tris++;
                if (PRIMARY) {
                    int4 vi = __ldg(pv.v4 + tl);
                    const Prim32 q = prim_test(__ldg(B.vview + vi.x), __ldg(B.vview + vi.y), __ldg(B.vview + vi.z), uc,
                                               vc, delta, B.w0_32);
                    if (!classify<COUNT>(q.U, q.V, q.W, q.eU, q.eV, q.eW, q.T, q.det, tlo, tau, p, tl, best, true, cn,
                                         cd)) {
                        clean = false;
                        sp = 0;
                    }
                } else {
                    const float4 *tr = pv.tri + (size_t)tl * 3;
                    float4 a = __ldg(tr), b = __ldg(tr + 1), c = __ldg(tr + 2);
                    if (__float_as_int(a.w) != skip) {
                        const Shear32 q = shear_test(r, a, b, c, delta);
                        // the common case first
                        if (certain_miss(q)) {
                            if (sp == 0) break;
                            ref = stack[--sp];
                            continue;
                        }
                        float eU, eV, eW;
                        shear_bounds(q, eU, eV, eW);
                        float det = q.U + q.V + q.W;
                        float T = fmaf(q.U, r.Sz * q.Akz, fmaf(q.V, r.Sz * q.Bkz, q.W * (r.Sz * q.Ckz)));
                        if (!classify<COUNT>(q.U, q.V, q.W, eU, eV, eW, T, det, tlo, tau, p, tl, best, false, cn, cd)) { clean = false; sp = 0; }
                    }
                }
            }
            // a handed-off ray (overflow) is re-traced from scratch: its stack was emptied
            if (sp == 0) break;
            ref = stack[--sp];
        }
    }
    if (COUNT) { cn.nodes += n_nodes; cn.tris += n_tris; cn.boxes += n_boxes; }
    return clean;
}

// The one-lane walk out of line (rare), where its registers do not weigh on the
// kernels that call it.
struct Near32 {
    Best32 b;
    Counts cn;
    int cand_n;
    int ok;
};

template <bool COUNT, bool COPY>
__device__ __noinline__ Near32 nearest32_primary(const TraceCtx &B, const Ray32 r, float uc, float vc, float delta,
                                                 float tau, Counts cn, Cands cd)
{
    Near32 o;
    o.ok = nearest32<COUNT, true, COPY>(B, r, uc, vc, 0.0f, -1, -1, kNoGroup, delta, tau, o.b, cn, cd) ? 1 : 0;
    o.cn = cn;
    o.cand_n = cd.n;
    return o;
}

template <bool COUNT>
__device__ __noinline__ Near32 nearest32_secondary(const TraceCtx &B, const Ray32 r, int skip, int gpart, int gskip,
                                                   float delta, float tau, Counts cn, Cands cd)
{
    Near32 o;
    o.ok = nearest32<COUNT, false, false>(B, r, 0.0f, 0.0f, B.eps32, skip, gpart, gskip, delta, tau, o.b, cn, cd) ? 1 : 0;
    o.cn = cn;
    o.cand_n = cd.n;
    return o;
}

// ------------------------------------------------------------- warp walk
// Two FP32 fused multiply-adds in one instruction, each rounded as fmaf.
__device__ __forceinline__ void ffma2(float &x, float &y, float a0, float a1, unsigned long long b, unsigned long long c)
{
    unsigned long long a, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(a0), "f"(a1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(d));
}
__device__ __forceinline__ unsigned long long pair2(float v)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float min3(float a, float b, float c)
{
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// The secondary segments of a warp's rays, walked together.  The open (ray,
// node) pairs of all 32 rays are in one list; a batch takes up to 32 of them, a
// lane a pair: the lane tests the node's four child boxes and appends those
// entered, nodes to the list and triangles to a second one, which is worked off
// 32 (ray, triangle) pairs at a time.  So every lane has work whatever the
// lengths of the rays' own walks, there is no per-ray stack, and a ray with a
// long walk is spread over the warp instead of holding it up.
//
// A walk by one lane (nearest32) goes from near to far and passes by what lies
// beyond the best hit so far.  Here nothing is passed by: the pairs come in no
// particular order until every triangle whose boxes the ray enters has been
// tested.  Nearly all are certain misses, which have no effect wherever they
// come.  The others are classified; when a ray's are all certain and no two
// distances (or the self-hit threshold) lie within the band of each other, the
// nearest one is the answer of the one-lane walk, bit for bit.  Otherwise what
// the one-lane walk makes of them depends on its order (which uncertain
// triangles it meets before it knows the hit in front of them), and the ray's
// few triangles are decided again in that order: walk_order finds a triangle's
// place in it from the sorted entry distances of the nodes above its leaf.
//
// What bounds it: a batch's chain of dependent fetches, tests and list updates,
// 1900-2650 cycles, against ~2700 for a step of 32 one-lane walks, which advances
// only the lanes whose rays are still walking.  It issues more instructions in
// all (nothing is culled, 10-20% more nodes; the lists), so a launch whose tiles
// fill the GPU many times over is faster with one-lane walks (headline batch 3.95
// against 5.97 ms): it is used where single walks are what a launch waits for
// (k_trace_few), and where rays are incoherent (k_diffuse: 8 evaluations of 50k
// triangles, 256^2, 16 samples a hit, 3.67 -> 3.08 ms).
constexpr int kNodeList = 256, kTriList = 160, kFound = 128;
struct WalkShared {  // of one warp
    float4 ra[32];   // origin, packed (part, node) of the origin's coplanar group
    float4 rb[32];   // 1 / direction, original id of the triangle left
    float4 rc[32];   // shear, code
    unsigned node[kNodeList];  // ray | part | node; after the walk the found triangles' distances and kinds, then the candidates
    unsigned tri[kTriList];    // ray | part | triangle
    unsigned found[kFound];    // ray | part | triangle: not a certain miss
};
static_assert(kNodeList >= 2 * kFound && kNodeList >= 32 * kCand, "reuse of the node list");

// Place of the leaf of triangle (p, tl) in the one-lane walk of ray r: key
// orders the leaves (the place of the part among the parts the ray enters, then
// per level the place of the child among its node's children, sorted as
// node4_step sorts them), pkey is the key of the leaf's node (what comes before
// it was decided when the node was opened), tn the entry distance of the leaf.
// Children beyond the best hit of the moment sort behind the others in the
// one-lane walk too, so leaving them in moves nothing.
__device__ __forceinline__ void walk_order(const TraceCtx &B, const float *o, const float *inv, float tlo, int p, int tl,
                                           const int *leaf_parent, unsigned long long &key, unsigned long long &pkey,
                                           float &tn)
{
    const float oi[3] = {o[0] * inv[0], o[1] * inv[1], o[2] * inv[2]};
    const int oct = (inv[0] < 0.f ? 1 : 0) | (inv[1] < 0.f ? 2 : 0) | (inv[2] < 0.f ? 4 : 0);
    int place = 0;
    float te = 0.0f;
    for (int q = -1; q < B.n_parts; q++) {  // the part's own distance first
        const float *box = B.part[q < 0 ? p : q].box_src;
        const float t = box_enter(box[0], box[3], box[1], box[4], box[2], box[5], inv, oi, tlo, INFINITY);
        if (q < 0) te = t;
        else if (t < te || (t == te && q < p)) place++;
    }
    tn = te;
    unsigned long long digits = 0ull;
    int depth = 0;
    const PartView &pv = B.part[p];
    const int ox = oct & 1, oy = (oct >> 1) & 1, oz = (oct >> 2) & 1;
    for (int up = __ldg(leaf_parent + pv.tri_begin + tl); up >= 0 && depth < kWalkDepth; depth++) {
        const float4 *nd = pv.node + (size_t)(up >> 2) * kNode4;
        const float4 nx = __ldg(nd + ox), fx = __ldg(nd + 1 - ox), ny = __ldg(nd + 2 + oy), fy = __ldg(nd + 3 - oy),
                     nz = __ldg(nd + 4 + oz), fz = __ldg(nd + 5 - oz);
        const int4 link = __ldg(reinterpret_cast<const int4 *>(nd + 7));
        float t[4];
        t[0] = box_enter_nf(nx.x, fx.x, ny.x, fy.x, nz.x, fz.x, inv, oi, tlo, INFINITY);
        t[1] = box_enter_nf(nx.y, fx.y, ny.y, fy.y, nz.y, fz.y, inv, oi, tlo, INFINITY);
        t[2] = box_enter_nf(nx.z, fx.z, ny.z, fy.z, nz.z, fz.z, inv, oi, tlo, INFINITY);
        t[3] = box_enter_nf(nx.w, fx.w, ny.w, fy.w, nz.w, fz.w, inv, oi, tlo, INFINITY);
        const int slot = up & 3;
        if (depth == 0) tn = slot == 0 ? t[0] : slot == 1 ? t[1] : slot == 2 ? t[2] : t[3];
        int c[4] = {0, 1, 2, 3};
        cswap(t[0], c[0], t[1], c[1]);
        cswap(t[2], c[2], t[3], c[3]);
        cswap(t[0], c[0], t[2], c[2]);
        cswap(t[1], c[1], t[3], c[3]);
        cswap(t[1], c[1], t[2], c[2]);
        const int at = c[0] == slot ? 0 : c[1] == slot ? 1 : c[2] == slot ? 2 : 3;
        digits |= (unsigned long long)at << (2 * depth);
        up = link.x < 0 ? -1 : ((link.x << 2) | link.y);
    }
    key = ((unsigned long long)place << 60) | (digits << (60 - 2 * depth));
    pkey = depth ? key & ~(3ull << (60 - 2 * depth)) : key;
}

// What a walk found, decided (out of line: fewer than half of the walks find
// anything, and its registers and code do not weigh on the walk).
struct WalkEnd {
    Best32 b;
    Counts cn;
    int cand_n;
    bool ok;
};
template <bool COUNT>
__device__ __noinline__ WalkEnd walk_settle(const TraceCtx &B, WalkShared &S, const MeshDev *mesh, bool live, bool over,
                                            int found, int gpart, int gskip, int skip, float delta, float tau, Counts cn)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u, nf = (unsigned)found;
    const float tlo = B.eps32, tnear = tlo - tau;
    const int rbits = B.ref_bits;
    const unsigned rmask = (1u << rbits) - 1u, pmask = (1u << (kWalkRefBits - rbits)) - 1u;
    Best32 best;
    best.t = INFINITY;
    best.part = -1;
    best.tl = -1;
    best.b1 = best.b2 = 0.0f;
    Cands cd;
    cd.n = 0;
    cd.id = reinterpret_cast<int *>(S.node) + lane;
    auto own = [&]() {
        const float4 A = S.ra[lane], C = S.rc[lane];
        return ShearRay{{A.x, A.y, A.z}, C.x, C.y, C.z, __float_as_int(C.w)};
    };
    // the one-lane walk, for the rays of lists that are full
    auto one_lane = [&]() {
        Ray32 r;
        const float4 A = S.ra[lane], I = S.rb[lane], C = S.rc[lane];
        const float o[3] = {A.x, A.y, A.z}, inv[3] = {I.x, I.y, I.z};
        for (int k = 0; k < 3; k++) { r.o[k] = o[k]; r.inv[k] = inv[k]; r.oi[k] = o[k] * inv[k]; r.d[k] = 0.0f; }
        r.Sx = C.x; r.Sy = C.y; r.Sz = C.z;
        r.code = __float_as_int(C.w);
        const Near32 w = nearest32_secondary<COUNT>(B, r, skip, gpart, gskip, delta, tau, cn, cd);
        best = w.b;
        cn = w.cn;
        cd.n = w.cand_n;
        return w.ok != 0;
    };
    bool ok = true;
    auto done = [&]() {
        __syncwarp();
        WalkEnd w;
        w.b = best;
        w.cn = cn;
        w.cand_n = cd.n;
        w.ok = ok;
        return w;
    };
    if (over) {
        if (live) ok = one_lane();
        return done();
    }
    // classify what was found, a lane each: distance and kind (0 nothing, 1 a
    // certain hit, 2 uncertain; + 4 where the plane distance of an uncertain one says something)
    float *fdist = reinterpret_cast<float *>(S.node);
    unsigned *fkind = S.node + kFound;
#pragma unroll 1
    for (unsigned f = (unsigned)lane; f < nf; f += 32u) {
        const unsigned e = S.found[f];
        const int ray = (int)(e >> 27);
        const float4 A = S.ra[ray], C = S.rc[ray];
        const ShearRay q = {{A.x, A.y, A.z}, C.x, C.y, C.z, __float_as_int(C.w)};
        const float4 *tr = B.part[(e >> rbits) & pmask].tri + (size_t)(e & rmask) * 3;
        const Shear32 t = shear_test(q, __ldg(tr), __ldg(tr + 1), __ldg(tr + 2), delta);
        float eU, eV, eW;
        shear_bounds(t, eU, eV, eW);
        const bool neg = (t.U < -eU) || (t.V < -eV) || (t.W < -eW), pos = (t.U > eU) || (t.V > eV) || (t.W > eW);
        const bool unsure = fabsf(t.U) <= eU || fabsf(t.V) <= eV || fabsf(t.W) <= eW;
        const float det = t.U + t.V + t.W;
        const float T = fmaf(t.U, q.Sz * t.Akz, fmaf(t.V, q.Sz * t.Bkz, t.W * (q.Sz * t.Ckz)));
        fdist[f] = T / det;
        fkind[f] = neg && pos ? 0u : (unsure ? (fabsf(det) > 1e-30f ? 6u : 2u) : 1u);
    }
    __syncwarp();
    // each ray's nearest certain hit, and what its certain hits' distances (d0 .. d3, ascending) leave open
    bool order = false;
    float d0 = INFINITY, d1 = INFINITY, d2 = INFINITY, d3 = INFINITY;
    unsigned hit = 0u, other = 0u;  // (other: one of its triangles is uncertain or in a tie)
#pragma unroll 1
    for (unsigned f = 0u; f < nf; f++) {
        if ((int)(S.found[f] >> 27) != lane) continue;
        const unsigned kind = fkind[f];
        const float t = fdist[f];
        if (kind == 1u) {
            if (fabsf(t - tlo) <= tau) other = 1u;
            else if (!(t > tlo)) continue;  // behind the origin: no effect
            else if (fabsf(t - d0) <= tau || fabsf(t - d1) <= tau || fabsf(t - d2) <= tau || fabsf(t - d3) <= tau ||
                     d3 < INFINITY)
                other = 1u;
            if (t > tlo) {
                if (t < d0) { d3 = d2; d2 = d1; d1 = d0; d0 = t; hit = S.found[f]; }
                else if (t < d1) { d3 = d2; d2 = d1; d1 = t; }
                else if (t < d2) { d3 = d2; d2 = t; }
                else if (t < d3) d3 = t;
            }
        } else if (kind != 0u && !((kind & 4u) && t < tnear)) {
            other = 1u;
        }
    }
    if (d0 < INFINITY) {
        best.part = (int)((hit >> rbits) & pmask);
        best.tl = (int)(hit & rmask);
        const float4 *tr = B.part[best.part].tri + (size_t)best.tl * 3;
        const Shear32 t = shear_test(own(), __ldg(tr), __ldg(tr + 1), __ldg(tr + 2), delta);
        const float id = 1.0f / (t.U + t.V + t.W);
        best.t = d0;
        best.b1 = t.V * id;
        best.b2 = t.W * id;
    }
    if (!__any_sync(kAll, other != 0u)) return done();
    // The rays with something open.  The one-lane walk meets every triangle whose
    // leaf is entered before the nearest certain hit plus its band, whatever its
    // order, and lists it when it is uncertain, or within the band of that hit or
    // of the self-hit threshold: such a ray's answer comes from the FP64
    // resolution, for which those triangles and the hit are enough (any others
    // that the one-lane walk lists lie beyond).  Only where what is open lies
    // beyond the nearest hit, or the lists would be near their end, does the
    // answer depend on the order.
    __syncwarp();
    bool sure = false;
    int n_sure = 0, n_far = 0;
    int *list = reinterpret_cast<int *>(S.tri);  // (a word per lane and round)
    for (unsigned f0 = 0u; f0 < nf; f0 += 32u) {
        // lane per triangle: is it open, and sure to be met?
        const unsigned f = f0 + (unsigned)lane;
        int what = 0;  // 1: sure to be listed, 2: open beyond the hit
        const int ray = f < nf ? (int)(S.found[f] >> 27) : 0;
        const float dr = __shfl_sync(kAll, d0, ray);
        const unsigned orr = __shfl_sync(kAll, other, ray);
        const unsigned hr = __shfl_sync(kAll, hit, ray);
        if (f < nf && orr) {
            const unsigned e = S.found[f], kind = fkind[f];
            const float t = fdist[f];
            const bool unsure = (kind & 2u) && !((kind & 4u) && t < tnear);
            const bool certain = kind == 1u && !(t < tnear && !(fabsf(t - tlo) <= tau));
            if (certain && e == hr) {
                what = fabsf(t - tlo) <= tau ? 1 : 0;
            } else if (unsure || certain) {
                // the leaf's box, as the refit forms it, and its entry distance
                const float4 A = S.ra[ray], I = S.rb[ray];
                const float inv[3] = {I.x, I.y, I.z}, oi[3] = {A.x * I.x, A.y * I.y, A.z * I.z};
                const float4 *tr = B.part[(e >> rbits) & pmask].tri + (size_t)(e & rmask) * 3;
                const float4 a = __ldg(tr), b = __ldg(tr + 1), c = __ldg(tr + 2);
                const float tn = box_enter(fminf(fminf(a.x, b.x), c.x) - B.pad, fmaxf(fmaxf(a.x, b.x), c.x) + B.pad,
                                           fminf(fminf(a.y, b.y), c.y) - B.pad, fmaxf(fmaxf(a.y, b.y), c.y) + B.pad,
                                           fminf(fminf(a.z, b.z), c.z) - B.pad, fmaxf(fmaxf(a.z, b.z), c.z) + B.pad, inv,
                                           oi, tnear, INFINITY);
                const bool met = tn <= dr + tau;
                if (unsure) what = met && (!(kind & 4u) || t <= dr + tau) ? 1 : 2;
                else if (met && (fabsf(t - tlo) <= tau || fabsf(t - dr) <= tau)) what = 1;
                else what = 3;  // a farther hit: open only in a tie with another one
            }
        }
        list[lane] = what;
        __syncwarp();
        // lane per ray again: its list
#pragma unroll 1
        for (unsigned g = 0u; g < 32u && f0 + g < nf; g++) {
            const unsigned e = S.found[f0 + g];
            if ((int)(e >> 27) != lane || !other) continue;
            const int w = list[g];
            if (w == 1) {
                sure = true;
                if (n_sure < 4) S.tri[32 * (1 + n_sure) + lane] = (((e >> rbits) & pmask) << 24) | (e & rmask);
                n_sure++;
            } else if (w != 0) {
                n_far++;
            }
        }
        __syncwarp();
    }
    // near the end of the list (the one-lane walk may list a hit that it drops later, too), the order decides
    order = other && (!sure || n_sure > 4 || 2 * n_sure + n_far > kCand);
    // (the node list's words are free from here for the rays that need no order)
    unsigned cs[4];
    for (int k = 0; k < 4; k++) cs[k] = other && !order && k < n_sure ? S.tri[32 * (1 + k) + lane] : 0u;
    __syncwarp();
    const unsigned om = __ballot_sync(kAll, order);
    auto listed = [&]() {
        if (other && !order)
            for (int k = 0; k < 4; k++)
                if (k < n_sure) push_cand(cd, (int)(cs[k] >> 24), (int)(cs[k] & 0xffffffu));
    };
    if (!om) {
        listed();
        return done();
    }
    if (order) {
        best.t = INFINITY;
        best.part = -1;
        best.tl = -1;
    }
    // the triangles of those rays, a lane each
    unsigned ne = 0u;
#pragma unroll 1
    for (unsigned f0 = 0u; f0 < nf; f0 += 32u) {
        const unsigned f = f0 + (unsigned)lane;
        const bool mine = f < nf && fkind[f] != 0u && ((om >> (S.found[f] >> 27)) & 1u);
        const unsigned m = __ballot_sync(kAll, mine);
        if (mine && ne + __popc(m & below) < 32u) S.tri[ne + __popc(m & below)] = f;
        ne += __popc(m);
    }
    __syncwarp();
    const bool mine = (unsigned)lane < min(ne, 32u);
    int ray = -1, id = 0;
    float t = 0.0f, tn = 0.0f;
    unsigned kind = 0u;
    unsigned long long key = ~0ull, pkey = ~0ull;
    if (mine) {
        const unsigned f = S.tri[lane], e = S.found[f];
        ray = (int)(e >> 27);
        id = (int)((((e >> rbits) & pmask) << 24) | (e & rmask));
        t = fdist[f];
        kind = fkind[f];
        const float4 A = S.ra[ray], I = S.rb[ray];
        const float o[3] = {A.x, A.y, A.z}, inv[3] = {I.x, I.y, I.z};
        walk_order(B, o, inv, tnear, id >> 24, id & 0xffffff, mesh->leaf_parent, key, pkey, tn);
    }
    __syncwarp();  // the node list's words are free now: they hold the candidates
    listed();
    if (ne > 32u) {
        if (order) ok = one_lane();
        return done();
    }
    // every such ray decides its triangles in the order of their keys, as
    // classify does; after: the best hit's distance once a lane's triangle was decided
    bool more = order;
    float after = INFINITY;
    unsigned long long last = 0ull;
    bool first = true;
    while (__any_sync(kAll, more)) {
        // the ray's next triangle
        unsigned long long next = ~0ull;
        int from = -1;
        for (int l = 0; l < (int)ne; l++) {  // (few)
            const unsigned long long k = __shfl_sync(kAll, key, l);
            const int rl = __shfl_sync(kAll, ray, l);
            if (rl == lane && (first || k > last) && (from < 0 || k < next)) { next = k; from = l; }
        }
        const int src = from < 0 ? 0 : from;
        const unsigned long long pk = __shfl_sync(kAll, pkey, src);
        const float lt = __shfl_sync(kAll, t, src), ltn = __shfl_sync(kAll, tn, src);
        const int lid = __shfl_sync(kAll, id, src);
        const unsigned lk = __shfl_sync(kAll, kind, src);
        // the best hit known when the leaf's node was opened: that after the last triangle before it
        float at_open = INFINITY;
        unsigned long long lastk = 0ull;
        bool any = false;
        for (int l = 0; l < (int)ne; l++) {  // (few)
            const unsigned long long k = __shfl_sync(kAll, key, l);
            const int rl = __shfl_sync(kAll, ray, l);
            const float al = __shfl_sync(kAll, after, l);
            if (rl == lane && k < pk && k < next && (!any || k > lastk)) { any = true; lastk = k; at_open = al; }
        }
        if (from < 0) more = false;
        if (more) {
            if (ltn <= at_open + tau) {
                if (lk & 2u) {
                    const bool far = (lk & 4u) && (lt > best.t + tau || lt < tlo - tau);
                    if (!far) {
                        if (COUNT) cn.why[1]++;
                        ok = push_cand(cd, lid >> 24, lid & 0xffffff);
                    }
                } else {
                    bool amb = false;
                    if (fabsf(lt - tlo) <= tau) { amb = true; if (COUNT) cn.why[3]++; }
                    else if (fabsf(lt - best.t) <= tau) { amb = true; if (COUNT) cn.why[2]++; }
                    if (amb) ok = push_cand(cd, lid >> 24, lid & 0xffffff);
                    if (ok && lt > tlo && lt < best.t) {
                        if (amb && best.part >= 0) ok = push_cand(cd, best.part, best.tl);
                        best.t = lt; best.part = lid >> 24; best.tl = lid & 0xffffff;
                    }
                }
            }
            if (!ok) more = false;  // handed off
            last = next;
            first = false;
        }
        // tell the lane of the triangle
        for (int l = 0; l < (int)ne; l++) {  // (few)
            const int who = __shfl_sync(kAll, ray, l);
            const int at = __shfl_sync(kAll, from, who);
            const float b = __shfl_sync(kAll, best.t, who);
            if (lane == l && at == l) after = b;
        }
    }
    if (order && ok && best.part >= 0) {
        const float4 *tr = B.part[best.part].tri + (size_t)best.tl * 3;
        const Shear32 q = shear_test(own(), __ldg(tr), __ldg(tr + 1), __ldg(tr + 2), delta);
        const float idet = 1.0f / (q.U + q.V + q.W);
        best.b1 = q.V * idet;
        best.b2 = q.W * idet;
    }
    return done();
}

// Nearest hits of a warp's secondary rays, a lane a ray (`live` where it has
// one); every lane calls it, with the segment's delta and tau.  best, cd and the
// result as nearest32 leaves them.
template <bool COUNT>
__device__ __forceinline__ bool walk_warp(const TraceCtx &B, WalkShared &S, const MeshDev *mesh, bool live, const Ray32 &r,
                                          int skip, int gpart, int gskip, float delta, float tau, Best32 &best,
                                          Counts &cn, Cands &cd)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float tlo = B.eps32, tnear = tlo - tau;
    const int rbits = B.ref_bits;
    const unsigned rmask = (1u << rbits) - 1u, pmask = (1u << (kWalkRefBits - rbits)) - 1u;
    best.t = INFINITY;
    best.part = -1;
    best.tl = -1;
    cd.n = 0;
    bool fall = rbits == 0;  // to the one-lane walk
    unsigned nn = 0u, nt = 0u, nf = 0u;  // entries of the three lists
    bool over = fall;                    // (uniform over the warp)
    // the group's packed part and node, or a value no entry has
    const unsigned gent = gskip == kNoGroup ? 0xffffffffu : ((unsigned)gpart << rbits) | (unsigned)gskip;
    if (live) {
        S.ra[lane] = make_float4(r.o[0], r.o[1], r.o[2], __uint_as_float(gent));
        S.rb[lane] = make_float4(r.inv[0], r.inv[1], r.inv[2], __int_as_float(skip));
        S.rc[lane] = make_float4(r.Sx, r.Sy, r.Sz, __int_as_float(r.code));
    }
    __syncwarp();
    if (!fall) {
        int part = 0;
        const int np = B.n_parts;
        int guard = B.walk_bound;
        while (true) {
            // the next parts' roots while there is room
            while (part < np && nn <= (unsigned)(kNodeList / 2 - 32) && nt < 32u) {
                const PartView &pv = B.part[part];
                const float *box = pv.box_src;
                bool in = false;
                if (live && !(part == gpart && pv.root == gskip))  // (else the whole part is the origin's plane)
                    in = box_enter(box[0], box[3], box[1], box[4], box[2], box[5], r.inv, r.oi, tnear, INFINITY) != INFINITY;
                const unsigned m = __ballot_sync(kAll, in);
                const unsigned e = ((unsigned)lane << 27) | ((unsigned)part << rbits);  // node 0 or triangle 0
                if (pv.root >= 0) {
                    if (in) S.node[nn + __popc(m & below)] = e;
                    nn += __popc(m);
                } else {
                    if (in) S.tri[nt + __popc(m & below)] = e;
                    nt += __popc(m);
                }
                part++;
            }
            __syncwarp();
            if (nn + nt == 0u) {
                if (part < np) continue;
                break;
            }
            if (--guard < 0) {
                if (live) cn.flags |= kFlagStack;
                return !live;
            }
            if (nt >= 32u || nn == 0u) {
                const unsigned m = min(nt, 32u);
                bool keep = false;
                unsigned e = 0u;
                if ((unsigned)lane < m) {
                    e = S.tri[nt - 1u - (unsigned)lane];
                    const int ray = (int)(e >> 27);
                    const float4 A = S.ra[ray], C = S.rc[ray];
                    const ShearRay q = {{A.x, A.y, A.z}, C.x, C.y, C.z, __float_as_int(C.w)};
                    const float4 *tr = B.part[(e >> rbits) & pmask].tri + (size_t)(e & rmask) * 3;
                    const float4 va = __ldg(tr), vb = __ldg(tr + 1), vc = __ldg(tr + 2);
                    keep = __float_as_int(va.w) != __float_as_int(S.rb[ray].w) &&
                           !certain_miss(shear_test(q, va, vb, vc, delta));
                    if (COUNT) cn.tris++;
                }
                nt -= m;
                const unsigned mk = __ballot_sync(kAll, keep);
                if (mk) {
                    const unsigned at = nf + __popc(mk & below);
                    if (keep && at < (unsigned)kFound) S.found[at] = e;
                    nf += __popc(mk);
                }
            } else {
                // a batch of nodes: as many as their children have room for; one at a time
                // at the end of the room, which is then a depth-first walk
                const int room = (kNodeList - B.walk_spare - (int)nn) / 3;
                const unsigned m = min(nn, (unsigned)min(32, max(room, 1)));
                bool in[4] = {false, false, false, false};
                int4 c = make_int4(0, 0, 0, 0);
                unsigned head = 0u, gent = 0u;
                if ((unsigned)lane < m) {
                    const unsigned e = S.node[nn - 1u - (unsigned)lane];
                    head = e & ~rmask;
                    const float4 A = S.ra[e >> 27], I = S.rb[e >> 27];
                    gent = __float_as_uint(A.w);
                    const int ox = I.x < 0.f ? 1 : 0, oy = I.y < 0.f ? 1 : 0, oz = I.z < 0.f ? 1 : 0;
                    const float4 *nd = B.part[(e >> rbits) & pmask].node + (size_t)(e & rmask) * kNode4;
                    const float4 nx = __ldg(nd + ox), fx = __ldg(nd + 1 - ox), ny = __ldg(nd + 2 + oy),
                                 fy = __ldg(nd + 3 - oy), nz = __ldg(nd + 4 + oz), fz = __ldg(nd + 5 - oz);
                    c = __ldg(reinterpret_cast<const int4 *>(nd + 6));
                    // the slab tests of box_enter_nf, two children at a time, nothing beyond to cull by
                    const unsigned long long ix = pair2(I.x), iy = pair2(I.y), iz = pair2(I.z);
                    const unsigned long long jx = pair2(-(A.x * I.x)), jy = pair2(-(A.y * I.y)), jz = pair2(-(A.z * I.z));
                    float x0, x1, y0, y1, z0, z1, X0, X1, Y0, Y1, Z0, Z1;
                    ffma2(x0, x1, nx.x, nx.y, ix, jx); ffma2(y0, y1, ny.x, ny.y, iy, jy); ffma2(z0, z1, nz.x, nz.y, iz, jz);
                    ffma2(X0, X1, fx.x, fx.y, ix, jx); ffma2(Y0, Y1, fy.x, fy.y, iy, jy); ffma2(Z0, Z1, fz.x, fz.y, iz, jz);
                    in[0] = max3(x0, y0, fmaxf(z0, tnear)) <= min3(X0, Y0, Z0);
                    in[1] = max3(x1, y1, fmaxf(z1, tnear)) <= min3(X1, Y1, Z1);
                    ffma2(x0, x1, nx.z, nx.w, ix, jx); ffma2(y0, y1, ny.z, ny.w, iy, jy); ffma2(z0, z1, nz.z, nz.w, iz, jz);
                    ffma2(X0, X1, fx.z, fx.w, ix, jx); ffma2(Y0, Y1, fy.z, fy.w, iy, jy); ffma2(Z0, Z1, fz.z, fz.w, iz, jz);
                    in[2] = max3(x0, y0, fmaxf(z0, tnear)) <= min3(X0, Y0, Z0);
                    in[3] = max3(x1, y1, fmaxf(z1, tnear)) <= min3(X1, Y1, Z1);
                    if (COUNT) { cn.nodes++; cn.boxes += 4; }
                }
                nn -= m;
                const unsigned hp = head & 0x07ffffffu;  // the part alone
                const int ck[4] = {c.x, c.y, c.z, c.w};
                bool inner[4], leaf[4];
                unsigned mi[4], ml[4];
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    leaf[k] = in[k] && ck[k] < 0;
                    inner[k] = in[k] && ck[k] >= 0 && (hp | (unsigned)ck[k]) != gent;
                    mi[k] = __ballot_sync(kAll, inner[k]);
                    ml[k] = __ballot_sync(kAll, leaf[k]);
                }
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    if (inner[k]) S.node[nn + __popc(mi[k] & below)] = head | (unsigned)ck[k];
                    if (leaf[k]) S.tri[nt + __popc(ml[k] & below)] = head | (unsigned)~ck[k];
                    nn += __popc(mi[k]);
                    nt += __popc(ml[k]);
                }
            }
            __syncwarp();
        }
        over = nf > (unsigned)kFound;
    }
    if (!over && nf == 0u) return true;
    const WalkEnd w = walk_settle<COUNT>(B, S, mesh, live, over, (int)nf, gpart, gskip, skip, delta, tau, cn);
    best = w.b;
    cn = w.cn;
    cd.n = w.cand_n;
    return w.ok;
}

// Compensated FP32 sums (the Kahan-Babuska form of compensated summation):
// the value is hi + lo, lo collecting the exact rounding error of every
// addition into hi (Knuth's TwoSum), so the sum keeps about twice FP32's
// precision without FP64 arithmetic.
struct Comp32 {
    float hi, lo;
};
__device__ __forceinline__ void comp_add(Comp32 &c, float x)
{
    const float s = __fadd_rn(c.hi, x);
    const float bp = __fsub_rn(s, c.hi);
    const float e = __fadd_rn(__fsub_rn(c.hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    c.hi = s;
    c.lo = __fadd_rn(c.lo, e);
}
__device__ __forceinline__ void comp_merge(Comp32 &c, const Comp32 &d)
{
    comp_add(c, d.hi);
    c.lo = __fadd_rn(c.lo, d.lo);
}
__device__ __forceinline__ float comp_value(const Comp32 &c) { return __fadd_rn(c.hi, c.lo); }

// Slot of flattened trace block g: the last slot whose first block is <= g.
__device__ __forceinline__ int slot_of_block(const SlotDesc *sd, int S, int g)
{
    int lo = 0, hi = S - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&sd[mid].tile0) <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __noinline__ Best32 resolve64_warp(const TraceCtx &B, bool want, int N, int i, int j, int seg, const int *hpt,
                                              int hps, int skip, Cands cd, Best32 best);
__device__ __noinline__ Best32 resolve64(const TraceCtx &B, int N, int i, int j, int seg, const int *hpt, int hps,
                                         int skip, Cands cd, Best32 best);

// ------------------------------------------------------------- raster
// Primary visibility by rasterisation.  Every primary ray of an evaluation runs
// along the same direction d from its pixel centre, so the nearest hit of a
// pixel is the nearest triangle whose view-frame projection covers the centre:
// each triangle visits the pixel centres of its projected box and applies the
// very test the traversal would (prim_test).  Pass 0 keeps, per pixel, the
// nearest certain hit (64-bit atomic minimum of depth bits and triangle).
// Pass 1 lists the pixel's triangles the FP32 test could not settle against
// that minimum: uncertain edge decisions not certainly beyond it, and certain
// hits within its depth band (what the traversal sends to its FP64
// resolution).  The trace then settles those candidates in FP64 exactly as
// after a traversal; a pixel with more than kPixMax of them traverses, and so does
// one with more than kPixCand where the slot's list ran over (pix_listed).

struct RastView {
    const float4 *vview;
    float umin32, vmin32, du32, dv32, rdu32, rdv32, w0, delta, tau;
    int N;
};

__device__ __forceinline__ RastView rast_view(const TraceArgs &a, int s)
{
    const TraceCtx *g = reinterpret_cast<const TraceCtx *>(a.tctx) + s;
    RastView V;
    V.vview = g->vview;
    V.umin32 = g->umin32; V.vmin32 = g->vmin32; V.du32 = g->du32; V.dv32 = g->dv32;
    V.rdu32 = g->rdu32; V.rdv32 = g->rdv32;
    V.w0 = g->w0_32; V.delta = g->delta_p; V.tau = g->tau_p;
    V.N = a.sd[s].N;
    return V;
}

// Pixels whose centre lies within the triangle's projected box widened by a
// hundredth of a pixel plus 64 delta: every other centre is outside the exact
// projection by more than the coordinate error, so the pixel cannot be hit.
__device__ __forceinline__ bool rast_box(const RastView &V, float4 a, float4 b, float4 c, int &i0, int &i1, int &j0,
                                         int &j1)
{
    const float mu = 0.01f * V.du32 + 64.0f * V.delta, mv = 0.01f * V.dv32 + 64.0f * V.delta;
    const float lim = (float)V.N + 1.0f;
    // products with the reciprocal pixel sizes: their rounding (~1e-4 pixel at
    // N = 1024) is far inside the hundredth of a pixel the box is widened by
    float ulo = (fminf(fminf(a.x, b.x), c.x) - mu - V.umin32) * V.rdu32 - 0.5f;
    float uhi = (fmaxf(fmaxf(a.x, b.x), c.x) + mu - V.umin32) * V.rdu32 - 0.5f;
    float vlo = (fminf(fminf(a.y, b.y), c.y) - mv - V.vmin32) * V.rdv32 - 0.5f;
    float vhi = (fmaxf(fmaxf(a.y, b.y), c.y) + mv - V.vmin32) * V.rdv32 - 0.5f;
    ulo = fminf(fmaxf(ulo, -1.0f), lim); uhi = fminf(fmaxf(uhi, -1.0f), lim);
    vlo = fminf(fmaxf(vlo, -1.0f), lim); vhi = fminf(fmaxf(vhi, -1.0f), lim);
    i0 = max((int)ceilf(ulo), 0); i1 = min((int)floorf(uhi), V.N - 1);
    j0 = max((int)ceilf(vlo), 0); j1 = min((int)floorf(vhi), V.N - 1);
    return i0 <= i1 && j0 <= j1;
}

// Can pixel centres [ib, ie] x [jb, je] meet the projected triangle?  False
// only when all four corners lie more than a pixel outside one edge line.
__device__ __forceinline__ bool chunk_meets(const RastView &V, float4 a, float4 b, float4 c, int ib, int ie, int jb,
                                            int je)
{
    const float u0 = fmaf((float)ib + 0.5f, V.du32, V.umin32), u1 = fmaf((float)ie + 0.5f, V.du32, V.umin32);
    const float v0 = fmaf((float)jb + 0.5f, V.dv32, V.vmin32), v1 = fmaf((float)je + 0.5f, V.dv32, V.vmin32);
    const float area = (b.x - a.x) * (c.y - a.y) - (b.y - a.y) * (c.x - a.x);
    const float pix = V.du32 + V.dv32;
    if (!(fabsf(area) > 1e-3f * pix * pix)) return true;  // sliver: keep every chunk
    const float sg = area > 0.0f ? 1.0f : -1.0f;
    const float px[3] = {a.x, b.x, c.x}, py[3] = {a.y, b.y, c.y};
    for (int e = 0; e < 3; e++) {
        const int f = e == 2 ? 0 : e + 1;
        const float ex = px[f] - px[e], ey = py[f] - py[e];
        const float m = pix * (fabsf(ex) + fabsf(ey));
        // edge function, positive inside: sg ((q - p) x (x - p))
        const float e00 = sg * (ex * (v0 - py[e]) - ey * (u0 - px[e]));
        const float e01 = sg * (ex * (v1 - py[e]) - ey * (u0 - px[e]));
        const float e10 = sg * (ex * (v0 - py[e]) - ey * (u1 - px[e]));
        const float e11 = sg * (ex * (v1 - py[e]) - ey * (u1 - px[e]));
        if (fmaxf(fmaxf(e00, e01), fmaxf(e10, e11)) < -m) return false;
    }
    return true;
}

// An upper bound, over the pixel centres [i0, i1] x [j0, j1], of the error
// bounds prim_test forms for the triangle: every coordinate relative to a
// centre is at most xm (u) or ym (v) in size, and FP32 rounding is monotone.
__device__ __forceinline__ float rast_bound(const RastView &V, float4 a, float4 b, float4 c, int i0, int i1, int j0,
                                            int j1)
{
    const float u0 = fmaf((float)i0 + 0.5f, V.du32, V.umin32), u1 = fmaf((float)i1 + 0.5f, V.du32, V.umin32);
    const float v0 = fmaf((float)j0 + 0.5f, V.dv32, V.vmin32), v1 = fmaf((float)j1 + 0.5f, V.dv32, V.vmin32);
    const float xm = fmaxf(fmaxf(fmaxf(fabsf(a.x - u0), fabsf(a.x - u1)), fmaxf(fabsf(b.x - u0), fabsf(b.x - u1))),
                           fmaxf(fabsf(c.x - u0), fabsf(c.x - u1)));
    const float ym = fmaxf(fmaxf(fmaxf(fabsf(a.y - v0), fabsf(a.y - v1)), fmaxf(fabsf(b.y - v0), fabsf(b.y - v1))),
                           fmaxf(fabsf(c.y - v0), fabsf(c.y - v1)));
    return (V.delta * (2.0f * xm + 2.0f * ym) + 4.0f * kU * (2.0f * xm * ym)) * 1.001f;
}

// The pixel key (one 64-bit word per pixel): the nearest certain hit's depth
// bits in the high word; in the low word a 3-bit field (bits 29-31) holding 7
// minus the number of uncertain candidates pass 1 listed (saturating at 7: more
// than kPixMax, the ray then traverses; the ones past kPixCand are in the slot's
// list of such) and the hit as part << 24 |
// part-local triangle (bits 0-27).  All ones: no certain hit, no candidate.
// Pass 0 writes its keys with the field at 7, so the 64-bit minimum orders by
// depth, then triangle; pass 1 only lowers the field.
static_assert(kMaxParts <= 16, "the pixel key holds the part in 4 bits");
constexpr unsigned kKeyId = 0x0fffffffu;
constexpr unsigned kKeyField = 29;
__device__ __forceinline__ bool key_none(unsigned long long k) { return (unsigned)(k >> 32) == 0xffffffffu; }
__device__ __forceinline__ unsigned key_cands(unsigned long long k) { return 7u - ((unsigned)(k >> kKeyField) & 7u); }

// Slot s's list of candidates past a pixel's first kPixCand: its length, a spare
// word, then (pixel, triangle) pairs; reset by the frame kernel.
__device__ __forceinline__ unsigned *slot_over(const TraceArgs &a, int s) { return a.pix_over + (size_t)s * kOverWords; }

// Are the pn candidates of a pixel all listed (else its ray traverses)?  Past
// kPixCand they are while the slot's list holds those of all its pixels: which
// entries a list that ran over has lost depends on the order of arrival, how many
// were counted does not, so such a list counts for none of the pixels.
__device__ __forceinline__ bool pix_listed(unsigned pn, const unsigned *over)
{
    return pn <= (unsigned)kPixCand || (pn <= (unsigned)kPixMax && __ldcg(over) <= (unsigned)kOverCap);
}

// A pixel's candidates past the first kPixCand into the ray's column (out of
// line: rare); returns how many candidates the column holds.
__device__ __noinline__ int over_cands(const unsigned *over, unsigned pix, int pn, int *col)
{
    const int n = (int)__ldcg(over);  // (pix_listed: at most kOverCap)
    int at = kPixCand;
    for (int k = 0; k < n; k++) {
        const uint2 e = __ldcg(reinterpret_cast<const uint2 *>(over) + 1 + k);
        if (e.x == pix && at < pn) col[at++ * kCandStride] = (int)e.y;
    }
    return at;
}

// One (triangle, pixel centre) pair.  E bounds the pair's error bounds: a
// decision certain against E is certain against them, so the exact bounds are
// formed only near an edge; the decisions are those of prim_test.
template <int PASS>
__device__ __forceinline__ void rast_pixel(const RastView &V, unsigned long long *key, unsigned *cand, unsigned *over, int i, int j,
                                           float4 a, float4 b, float4 c, unsigned id, float E)
{
    const float uc = fmaf((float)i + 0.5f, V.du32, V.umin32);
    const float vc = fmaf((float)j + 0.5f, V.dv32, V.vmin32);
    Prim32 q = prim_core(a, b, c, uc, vc, V.w0);
    if (((q.U < -E) || (q.V < -E) || (q.W < -E)) && ((q.U > E) || (q.V > E) || (q.W > E))) return;
    bool unsure = false;
    if (!(fabsf(q.U) > E && fabsf(q.V) > E && fabsf(q.W) > E)) {
        q = prim_test(a, b, c, uc, vc, V.delta, V.w0);
        const bool neg = (q.U < -q.eU) || (q.V < -q.eV) || (q.W < -q.eW);
        const bool pos = (q.U > q.eU) || (q.V > q.eV) || (q.W > q.eW);
        if (neg && pos) return;  // certainly outside
        unsure = fabsf(q.U) <= q.eU || fabsf(q.V) <= q.eV || fabsf(q.W) <= q.eW;
    }
    const float t = q.T / q.det;
    const size_t px = (size_t)i * V.N + j;
    if (PASS == 0) {
        // primary rays start at the window (tlo = 0); t > 0 orders as its bits
        if (!unsure && t > 0.0f)
            atomicMin(key + px, ((unsigned long long)__float_as_uint(t) << 32) | (7u << kKeyField) | id);
        return;
    }
    // (other pass-1 threads may lower this key's candidate field meanwhile:
    // depth and triangle stay as pass 0 left them)
    const unsigned long long k = key[px];
    const float tmin = key_none(k) ? INFINITY : __uint_as_float((unsigned)(k >> 32));
    bool take;
    if (unsure) take = !(fabsf(q.det) > 1e-30f && (t > tmin + V.tau || t < -V.tau));
    else take = fabsf(t) <= V.tau || (((unsigned)k & kKeyId) != id && fabsf(t - tmin) <= V.tau);
    if (take) {
        // claim a candidate slot by lowering the key's field; every failed
        // compare-and-swap means another thread's succeeded, and the loop is
        // bounded all the same: past the bound the field is cleared, which
        // sends the ray to the traversal (always correct)
        unsigned long long old = k;
        int slot = kPixMax;
        for (int it = 0; it < 64; it++) {
            const unsigned f = (unsigned)(old >> kKeyField) & 7u;
            if (f == 0u) break;  // saturated: the ray traverses
            const unsigned long long seen = atomicCAS(key + px, old, old - (1ull << kKeyField));
            if (seen == old) { slot = (int)(7u - f); break; }
            old = seen;
            if (it == 63) atomicAnd(key + px, ~(7ull << kKeyField));
        }
        if (slot < kPixCand) {
            cand[px * kPixCand + slot] = id;
        } else if (slot < kPixMax) {
            // a pixel on a vertex shared by several triangles (rare): the slot's own list of such
            // (counted past its end too: see pix_listed)
            const unsigned at = atomicAdd(over, 1u);
            if (at < (unsigned)kOverCap) reinterpret_cast<uint2 *>(over)[1 + at] = make_uint2((unsigned)px, id);
        }
    }
}

__device__ __forceinline__ int part_of_sorted(const MeshDev *m, int t)
{
    int p = 0;
    for (int q = 0; q < m->n_parts; q++)
        if (t >= m->part[q].tri_begin && t < m->part[q].tri_begin + m->part[q].tri_count) p = q;
    return p;
}

// Thread per (slot, sorted triangle): small projected boxes in place; larger
// ones are listed for k_raster_chunks, which lists their 16 x 16-pixel chunks
// that can meet them for k_raster_big (pass 0 lists, pass 1 reuses the lists).
template <int PASS>
__device__ __forceinline__ void raster_tri(const TraceArgs &a, int s, int t)
{
    const TraceCtx *g = reinterpret_cast<const TraceCtx *>(a.tctx) + s;
    // the slot's context in one round of loads (nothing read from the mesh record)
    const int skip = g->skip, n_tris = g->n_tris;
    const int4 *tv4 = g->tri_v4;
    const RastView V = rast_view(a, s);
    if (skip || t >= n_tris) return;
    if (!(V.du32 > 0.0f && V.dv32 > 0.0f)) {
        if (PASS == 0 && t == 0) a.rast_bad[s] = 1;
        return;
    }
    const int4 vi = __ldg(tv4 + t);
    const float4 A = __ldg(V.vview + vi.x), B = __ldg(V.vview + vi.y), C = __ldg(V.vview + vi.z);
    int i0, i1, j0, j1;
    if (!rast_box(V, A, B, C, i0, i1, j0, j1)) return;
    const int w = i1 - i0 + 1, h = j1 - j0 + 1;
    if (w * h > kRastSmall) {
        if (PASS == 0) {
            // listed for k_raster_chunks, which lists its chunks
            const unsigned at = atomicAdd(a.bigt_count, 1u);
            if (at >= (unsigned)a.big_cap) {
                a.rast_bad[s] = 1;
                return;
            }
            a.bigt[at] = make_int2(s, t);
        }
        return;
    }
    const unsigned id = (unsigned)vi.w;  // (part << 24) | index within the part
    const size_t off = (size_t)s * a.ray_stride;
    const float eb = rast_bound(V, A, B, C, i0, i1, j0, j1);
    for (int i = i0; i <= i1; i++)
        for (int j = j0; j <= j1; j++)
            rast_pixel<PASS>(V, a.pix_key + off, a.pix_cand + off * kPixCand, slot_over(a, s), i, j, A, B, C, id, eb);
}

template <int PASS>
__global__ void __launch_bounds__(128) k_raster(TraceArgs a)
{
    pdl_enter();
    raster_tri<PASS>(a, blockIdx.y, blockIdx.x * blockDim.x + threadIdx.x);
}

// Warp per listed large triangle: its 16 x 16-pixel chunks that can meet it,
// tested a chunk per lane and appended with one atomic per warp pass.
__global__ void __launch_bounds__(256) k_raster_chunks(TraceArgs a)
{
    pdl_enter();
    const unsigned n = min(__ldcg(a.bigt_count), (unsigned)a.big_cap);
    const unsigned lane = threadIdx.x & 31u, nw = gridDim.x * (blockDim.x >> 5);
    for (unsigned e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < n; e += nw) {
        const int2 E = a.bigt[e];
        const int s = E.x, t = E.y;
        const TraceCtx *g = reinterpret_cast<const TraceCtx *>(a.tctx) + s;
        const int4 *tv4 = g->tri_v4;
        const RastView V = rast_view(a, s);
        const int4 vi = __ldg(tv4 + t);
        const float4 A = __ldg(V.vview + vi.x), B = __ldg(V.vview + vi.y), C = __ldg(V.vview + vi.z);
        int i0, i1, j0, j1;
        if (!rast_box(V, A, B, C, i0, i1, j0, j1)) continue;
        const int cw = (i1 - i0 + kRastChunk) / kRastChunk, ch = (j1 - j0 + kRastChunk) / kRastChunk;
        for (int k0 = 0; k0 < cw * ch; k0 += 32) {
            const int k = k0 + (int)lane;
            bool meets = false;
            if (k < cw * ch) {
                const int ib = i0 + (k % cw) * kRastChunk, jb = j0 + (k / cw) * kRastChunk;
                meets = chunk_meets(V, A, B, C, ib, min(ib + kRastChunk - 1, i1), jb, min(jb + kRastChunk - 1, j1));
            }
            const unsigned bal = __ballot_sync(0xffffffffu, meets);
            if (!bal) continue;
            unsigned at = 0u;
            if (lane == 0) at = atomicAdd(a.big_count, (unsigned)__popc(bal));
            at = __shfl_sync(0xffffffffu, at, 0);
            const unsigned cnt = (unsigned)__popc(bal);
            const unsigned room = at < (unsigned)a.big_cap ? (unsigned)a.big_cap - at : 0u;
            if (cnt > room) {
                // the list is full: the slot's pixels traverse instead; the part of this
                // warp's range below the capacity is filled with placeholders (slot -1)
                // so that every entry a reader sees was written
                const unsigned idx = at + __popc(bal & ((1u << lane) - 1u));
                if (meets && idx < (unsigned)a.big_cap) a.big[idx] = make_int4(-1, 0, 0, 0);
                if (lane == 0) a.rast_bad[s] = 1;
                break;
            }
            if (meets) a.big[at + __popc(bal & ((1u << lane) - 1u))] = make_int4(s, t, k % cw, k / cw);
            if (a.queue && lane == 0) atomicAdd(a.qstate + kQSlot + 3 * s + 2, cnt);
        }
    }
}

// One listed chunk of a large triangle, by the calling warp.  Returns the
// entry's slot, or -1 for a placeholder of a full list.
template <int PASS>
__device__ __forceinline__ int raster_big_entry(const TraceArgs &a, unsigned e, unsigned lane)
{
    const int4 E = a.big[e];
    const int s = E.x, t = E.y;
    if (s < 0) return -1;
    const TraceCtx *g = reinterpret_cast<const TraceCtx *>(a.tctx) + s;
    const int4 *tv4 = g->tri_v4;
    const RastView V = rast_view(a, s);
    const int4 vi = __ldg(tv4 + t);
    const float4 A = __ldg(V.vview + vi.x), B = __ldg(V.vview + vi.y), C = __ldg(V.vview + vi.z);
    int i0, i1, j0, j1;
    if (!rast_box(V, A, B, C, i0, i1, j0, j1)) return s;
    const int ib = i0 + E.z * kRastChunk, jb = j0 + E.w * kRastChunk;
    const int ie = min(ib + kRastChunk - 1, i1), je = min(jb + kRastChunk - 1, j1);
    const unsigned id = (unsigned)vi.w;  // (part << 24) | index within the part
    const size_t off = (size_t)s * a.ray_stride;
    const float eb = rast_bound(V, A, B, C, ib, ie, jb, je);
    for (int q = (int)lane; q < kRastChunk * kRastChunk; q += 32) {
        const int i = ib + q / kRastChunk, j = jb + q % kRastChunk;
        if (i <= ie && j <= je)
            rast_pixel<PASS>(V, a.pix_key + off, a.pix_cand + off * kPixCand, slot_over(a, s), i, j, A, B, C, id, eb);
    }
    return s;
}

// Warp per listed chunk of a large triangle (grid-stride over the list).
template <int PASS>
__global__ void __launch_bounds__(256) k_raster_big(TraceArgs a)
{
    pdl_enter();
    const unsigned n = min(__ldcg(a.big_count), (unsigned)a.big_cap);
    const unsigned lane = threadIdx.x & 31u, nw = gridDim.x * (blockDim.x >> 5);
    for (unsigned e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < n; e += nw) raster_big_entry<PASS>(a, e, lane);
}

// The second raster pass in one launch: blocks below nbig take listed chunks
// of large triangles (a warp per chunk, grid-stride over the list), the rest a
// small triangle per thread (per_slot blocks a slot).
__global__ void __launch_bounds__(128) k_raster_pass1(TraceArgs a, int nbig, int per_slot)
{
    pdl_enter();
    if ((int)blockIdx.x < nbig) {
        const unsigned n = min(__ldcg(a.big_count), (unsigned)a.big_cap);
        const unsigned lane = threadIdx.x & 31u, nw = (unsigned)nbig * (blockDim.x >> 5);
        for (unsigned e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < n; e += nw) raster_big_entry<1>(a, e, lane);
        return;
    }
    const int b = (int)blockIdx.x - nbig;
    raster_tri<1>(a, b / per_slot, (b % per_slot) * (int)blockDim.x + (int)threadIdx.x);
}

// Momentum of one hit of direction d and weight wgt: f = w [(1 - rho_s) d - 2
// (rho_s c + rho_d / 3) n_f], n_f = sg n, added with its torque about c_ref to
// acc.  Returns the hit point from the barycentric weights on the hit triangle
// (its error is that of the test, not that of a long FP32 ray), the unit
// normal, d . n, the specular coefficient and the original triangle id.
struct Shade32 {
    float hp[3], n[3], dn, rs;
    int orig;
};
__device__ __forceinline__ Shade32 shade_hit(const TraceCtx &B, const Best32 &h, const float *d, float wgt, float *acc)
{
    Shade32 o;
    const float4 *tr = B.part[h.part].tri + (size_t)h.tl * 3;
    float4 a0 = __ldg(tr), a1 = __ldg(tr + 1), a2 = __ldg(tr + 2);
    o.orig = __float_as_int(a0.w);
    unsigned mt = __float_as_uint(a1.w);
    float e1[3] = {a1.x - a0.x, a1.y - a0.y, a1.z - a0.z};
    float e2[3] = {a2.x - a0.x, a2.y - a0.y, a2.z - a0.z};
    float n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
    float il = rsqrtf(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    n[0] *= il; n[1] *= il; n[2] *= il;
    float dn = d[0] * n[0] + d[1] * n[1] + d[2] * n[2];
    int side = dn < 0.f ? 0 : 1;
    float sg = side ? -1.f : 1.f;
    float2 m = __ldg(B.mat32 + (side ? (mt >> 16) : (mt & 0xffffu)));
    float c = -sg * dn;
    float ka = wgt * (1.0f - m.x), kn = -2.0f * wgt * (m.x * c + m.y * (1.0f / 3.0f)) * sg;
    float F[3], arm[3];
    const float a0v[3] = {a0.x, a0.y, a0.z};
    for (int k = 0; k < 3; k++) {
        F[k] = ka * d[k] + kn * n[k];
        o.hp[k] = fmaf(h.b1, e1[k], fmaf(h.b2, e2[k], a0v[k]));
        arm[k] = o.hp[k] - B.cref32[k];
        o.n[k] = n[k];
    }
    acc[0] += F[0]; acc[1] += F[1]; acc[2] += F[2];
    acc[3] += arm[1] * F[2] - arm[2] * F[1];
    acc[4] += arm[2] * F[0] - arm[0] * F[2];
    acc[5] += arm[0] * F[1] - arm[1] * F[0];
    o.dn = dn;
    o.rs = m.x;
    return o;
}

// A triangle whose edges' cross product, or its square, underflows in FP32 (a sliver of 1e-23 m^2, or
// vertices that round to one line) has no FP32 normal: the ray goes to the FP64 re-trace, which has one.
__device__ __forceinline__ bool no_normal(const Shade32 &s) { return !(fabsf(s.dn) < 2.0f); }

// What a tile's 32 rays leave, by one warp, a lane a ray: the list of the rays
// handed to the FP64 path, force and torque, counts.
template <bool COUNT>
__device__ __forceinline__ void tile_results(const TraceArgs &a, int s, int tile_id, int ray, const float *fac,
                                             unsigned c_handoff, unsigned c_segs, unsigned c_hitbits, const Counts &cn,
                                             int flags)
{
    const int lane = threadIdx.x & 31;
    // tile-ordered list of the rays handed to the FP64 path
    const size_t tile = (size_t)s * a.n_blocks_x + tile_id;
    unsigned bal = __ballot_sync(0xffffffffu, c_handoff != 0u);
    if (c_handoff) a.amb_list[tile * kTileRays + __popc(bal & ((1u << lane) - 1u))] = ray;
    // tile sums, one partial per tile: force and torque by a fixed FP32
    // butterfly over the 32 rays (FP64 shuffles would occupy GB300's slow FP64
    // pipe), counts by integer reductions; every sum above the tile is FP64
    for (int k = 0; k < 6; k++) {
        float x = fac[k];
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) a.partials[tile * 6 + k] = x;
    }
    // counts 0..6 always (hand-offs, segments, hits per segment level); the
    // traversal counters only in the counting variant
#pragma unroll
    for (int k = 0; k < (COUNT ? kCnt : kCntRay); k++) {
        unsigned v;
        if (k == 0) v = c_handoff;
        else if (k == 1) v = c_segs;
        else if (k <= 2 + kMaxBounces) v = (c_hitbits >> (k - 2)) & 1u;
        else if (k == 7) v = cn.nodes;
        else if (k == 8) v = cn.tris;
        else if (k == 9) v = cn.boxes;
        else v = cn.why[k - 10];
        const unsigned x = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) a.pcounts[tile * kCnt + k] = x;
    }
    int fl = __reduce_or_sync(0xffffffffu, flags);
    if (lane == 0) {
        a.amb_count[tile] = __popc(bal);
        if (fl) atomicOr(&a.pose[s].flags, fl);
    }
}

// A block is kTraceWarps warps over consecutive tiles of one slot, sharing
// one copy of the slot's context; a warp past the slot's last tile idles.
// The trace of flattened block vb (kTraceWarps tiles of one slot).  B, s_cand
// and s_hpt are the block's shared context copy and per-thread columns (entry k
// of thread x at [k * kLaneStride + x]): the candidates of the FP64 resolution,
// and each segment's hit as (part, triangle) for the FP64 replay of the
// specular chain and the hit record.  QUEUE: run inside the work queue, where
// this SM may hold stale L1 copies of pixel keys another SM's second raster
// pass has changed since, so the raster's results are read from L2.
template <bool COUNT, bool HITS, bool QUEUE>
__device__ __forceinline__ void trace_block(const TraceArgs &a, int vb, TraceCtx &B, int *s_cand, int *s_hpt)
{
    static_assert(kTileRays * kTraceWarps == kLaneStride, "per-thread shared columns assume 128 threads");
    const int s = slot_of_block(a.sd, a.n_slots, vb);
    const SlotDesc &D = a.sd[s];
    const int tile_id = (vb - D.tile0) * kTraceWarps + (int)(threadIdx.x >> 5);
    const int N = D.N, nseg = D.nseg;
    const int lane = threadIdx.x & 31;
    const int tw = D.tile_w, lw = __ffs(tw) - 1;
    const int i = (tile_id % D.tiles_x) * tw + (lane & (tw - 1));
    const int j = (tile_id / D.tiles_x) * (kTileRays >> lw) + (lane >> lw);
    const bool inside = tile_id < D.tiles && i < N && j < N;
    // rasterised primary visibility of this pixel
    unsigned long long pk = ~0ull;
    bool bad = true;
    if (a.raster) {
        bad = a.rast_bad[s] != 0;
        const unsigned long long *key = a.pix_key + (size_t)s * a.ray_stride + (size_t)i * N + j;
        if (inside) pk = QUEUE ? __ldcg(key) : __ldcs(key);
    }
    // a block without a hit or candidate (half of a window's blocks) leaves before it copies the context
    // (its warps held their slots for ~10k cycles each: headline batch 3.95 -> 3.89 ms, 100k triangles at 777^2 2.57 ->
    // 2.51 ms, box-wing table 1.61 -> 1.57 ms; what the key read keeps alive across the copy spills: 49.0 -> 55.1 M
    // local-memory load sectors a headline launch)
    if (!__syncthreads_or(inside && (bad || pk != ~0ull))) {
        if (tile_id >= D.tiles) return;
        const size_t tile = (size_t)s * a.n_blocks_x + tile_id;
        const unsigned n = (unsigned)__popc(__ballot_sync(0xffffffffu, inside));
        if (lane == 0) a.amb_count[tile] = 0;
        const int skip = reinterpret_cast<const TraceCtx *>(a.tctx)[s].skip;
        if (skip == kSkipDist) return;
        if (HITS && inside) {
            int32_t *hq = a.hits + ((size_t)s * a.ray_stride + (size_t)i * N + j) * a.seg_stride;
            for (int k = 0; k < nseg; k++) hq[k] = -1;
        }
        if (skip) return;
        if (lane < 6) a.partials[tile * 6 + lane] = 0.0f;
        if (lane < (COUNT ? kCnt : kCntRay)) a.pcounts[tile * kCnt + lane] = lane == 1 ? n : 0u;  // (segments)
        return;
    }
    load_ctx(B, a, s);
    __syncthreads();
    if (tile_id >= D.tiles) return;
    if (B.skip) {
        if (lane == 0) a.amb_count[(size_t)s * a.n_blocks_x + tile_id] = 0;
        if (HITS && inside && B.skip == kSkipDir) {
            int32_t *hq = a.hits + ((size_t)s * a.ray_stride + (size_t)i * N + j) * a.seg_stride;
            for (int k = 0; k < nseg; k++) hq[k] = -1;
        }
        return;
    }
    // per-ray results: force / torque in FP32 (at most 1 + bounces terms); counts
    // as scalars (a hand-off flag, the segments traced, a bit per segment hit)
    float fac[6] = {0, 0, 0, 0, 0, 0};
    unsigned c_handoff = 0u, c_segs = 0u, c_hitbits = 0u;
    int flags = 0;
    const int ray = i * N + j;
    int *hpt = s_hpt + threadIdx.x;
    Counts cn = {0u, 0u, 0u, {0u, 0u, 0u, 0u}, 0};
    if (inside) {
        Ray32 r;
        for (int k = 0; k < 3; k++) r.d[k] = B.dir[k];
        const float uc = fmaf((float)i + 0.5f, B.du32, B.umin32);
        const float vc = fmaf((float)j + 0.5f, B.dv32, B.vmin32);
        float wgt = 1.0f;
        int skip = -1, gpart = -1, gskip = kNoGroup;
        float acc[6] = {0, 0, 0, 0, 0, 0};
        unsigned hitbits = 0u;
        bool clean = true;
        int nseg_done = 0;
        Cands cd;
        cd.n = 0;
        cd.id = s_cand + (threadIdx.x >> 5) * (kCand * kCandStride) + lane;
        float delta = B.delta_p, tau = B.tau_p;
        bool rast = false;
        if (a.raster) {
            const size_t px = (size_t)s * a.ray_stride + ray;
            const unsigned pn = key_cands(pk);
            rast = !bad && pix_listed(pn, slot_over(a, s));
            if (rast) {
                cd.n = (int)pn;
                for (int c = 0; c < min((int)pn, kPixCand); c++)
                    cd.id[c * kCandStride] = (int)(QUEUE ? __ldcg(a.pix_cand + px * kPixCand + c) : a.pix_cand[px * kPixCand + c]);
                if (pn > (unsigned)kPixCand) cd.n = over_cands(slot_over(a, s), (unsigned)ray, (int)pn, cd.id);
                if (COUNT) cn.why[0] += pn;
            }
        }
        for (int seg = 0; seg < nseg; seg++) {
            Best32 h;
            float tlo = seg == 0 ? 0.0f : B.eps32;
            nseg_done++;
            if (seg == 0 && !rast)  // a traversed primary segment starts at its pixel on the window
                for (int k = 0; k < 3; k++) r.o[k] = fmaf((float)i + 0.5f, B.du[k], fmaf((float)j + 0.5f, B.dv[k], B.org[k]));
            if (seg > 0 || !rast) ray_setup(r);  // the raster's primary segment needs no ray frame
            if (seg == 0 && rast) {
                // the raster's nearest certain hit; its barycentric weights as the traversal forms them
                h.t = INFINITY;
                h.part = -1;
                h.tl = -1;
                if (!key_none(pk)) {
                    const unsigned id = (unsigned)pk & kKeyId;
                    h.part = (int)(id >> 24);
                    h.tl = (int)(id & 0xffffffu);
                    const int4 vi = __ldg(B.part[h.part].v4 + h.tl);
                    const Prim32 q = prim_core(__ldg(B.vview + vi.x), __ldg(B.vview + vi.y), __ldg(B.vview + vi.z), uc,
                                               vc, B.w0_32);
                    const float id32 = 1.0f / q.det;
                    h.t = q.T * id32;  // not used past this point; the weights are the traversal's
                    h.b1 = q.V * id32;
                    h.b2 = q.W * id32;
                }
            } else {
                bool ok;
                if (seg == 0) {
                    const Near32 o = nearest32_primary<COUNT, true>(B, r, uc, vc, delta, tau, cn, cd);
                    h = o.b;
                    cn = o.cn;
                    cd.n = o.cand_n;
                    ok = o.ok != 0;
                } else {
                    ok = nearest32<COUNT, false, true>(B, r, uc, vc, tlo, skip, gpart, gskip, delta, tau, h, cn, cd);
                }
                if (!ok) {
                    clean = false;
                    break;
                }
            }
            if (cd.n > 0) h = resolve64(B, N, i, j, seg, hpt, kLaneStride, skip, cd, h);  // rare: settle in FP64
            if (h.part < 0) break;
            hpt[seg * kLaneStride] = (h.part << 24) | h.tl;
            hitbits |= 1u << seg;
            const Shade32 sh = shade_hit(B, h, r.d, wgt, acc);
            if (no_normal(sh)) { clean = false; break; }
            wgt *= sh.rs;
            if (seg + 1 >= nseg || wgt == 0.0f) break;
            for (int k = 0; k < 3; k++) {
                r.o[k] = sh.hp[k];
                r.d[k] = r.d[k] - 2.0f * sh.dn * sh.n[k];
            }
            skip = sh.orig;
            // the reflected ray leaves the hit triangle's plane at |dn|: its coplanar group can
            // only be met within dev / |dn| of the origin, inside the self-hit distance eps
            const int2 g = __ldg(B.grp + B.part[h.part].tri_begin + h.tl);
            gpart = h.part;
            gskip = fabsf(sh.dn) * B.eps32 > 16.0f * __int_as_float(g.y) ? g.x : kNoGroup;
            // next segment: world-frame test; the origin error grows with the previous bound
            delta = B.delta_s + 2.0f * delta;
            tau = 64.0f * delta + 32.0f * kU * (B.R + B.L);
        }
        flags = cn.flags;
        if (clean) {
            for (int k = 0; k < 6; k++) fac[k] = acc[k];
            c_segs = nseg_done;
            c_hitbits = hitbits;
            if (HITS) {
                int32_t *hq = a.hits + ((size_t)s * a.ray_stride + ray) * a.seg_stride;
                for (int k = 0; k < nseg; k++) {
                    int o = -1;
                    if ((hitbits >> k) & 1u) {
                        const int hk = hpt[k * kLaneStride];
                        o = __float_as_int(__ldg(B.part[hk >> 24].tri + (size_t)(hk & 0xffffff) * 3).w);
                    }
                    hq[k] = o;
                }
            }
        } else {
            c_handoff = 1u;
        }
    }
    tile_results<COUNT>(a, s, tile_id, ray, fac, c_handoff, c_segs, c_hitbits, cn, flags);
}

// 64 registers for 32 warps an SM (212 B of spill stores and 232 B of loads; 80 registers and fewer warps: slower).
template <bool COUNT, bool HITS>
__global__ void __launch_bounds__(kTileRays * kTraceWarps, 32 / kTraceWarps) k_trace(TraceArgs a)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char s_dyn[];
    TraceCtx &B = *reinterpret_cast<TraceCtx *>(s_dyn);
    int *s_hpt = reinterpret_cast<int *>(s_dyn + trace_ctx_dyn_bytes(a.ctx_parts));
    __shared__ int s_cand[kCand * kLaneStride];
    trace_block<COUNT, HITS, false>(a, blockIdx.x, B, s_cand, s_hpt);
}

// ------------------------------------------------------- few slots
// The trace of a launch of few slots (one evaluation of a propagation stage, a
// single call): a block is one tile.  Such a launch lasts as long as its
// slowest warps: the rays that go far lie together (a dish, a wing seen along
// its plane), and a warp with a lane per ray takes up to 200 us for such a tile
// while the launch's average SM is busy for 40.  Here the block's first warp, a
// lane a ray, takes the raster's results, shades and reflects; the rays that go
// on are dealt to the block's warps, and each walks its share together with all
// 32 lanes (walk_warp).  In launches of many slots the other
// slots' tiles fill the SMs meanwhile and the one-lane walks, which issue fewer
// instructions, are the faster ones.  More than half of a window's tiles are
// empty: their blocks read 32 keys and leave; the others read the slot's context
// in place (L1) instead of copying it first.
struct FewShared {  // of a block; entry of the ray's lane of the tile
    float4 ra[kTileRays], rb[kTileRays], rc[kTileRays];  // a ray that goes on: origin, skip; 1 / direction, gpart; shear, code
    float d[3][kTileRays], acc[6][kTileRays];
    int gskip[kTileRays];
    int res[kTileRays];                // its hit (part << 24 | triangle), -1 none, -2 handed off
    float b1[kTileRays], b2[kTileRays];
    int list[kTileRays];               // the lanes of the rays that go on
    int n_list, flags;
    int hpt[kMaxBounces + 1][kTileRays];
};
static_assert(kTileRays == kCandStride, "the hit columns have the stride of the candidates");

template <bool HITS>
__global__ void __launch_bounds__(32 * kFewWarps, kFewBlocksPerSM) k_trace_few(TraceArgs a)
{
    pdl_enter();
    __shared__ __align__(16) WalkShared s_walk[kFewWarps];
    __shared__ __align__(16) FewShared F;
    const int w = (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    // the slot: the launch's blocks are the slots' tiles end to end
    int s = 0, tile_id = (int)blockIdx.x;
    while (s + 1 < a.n_slots && tile_id >= a.sd[s].tiles) tile_id -= a.sd[s++].tiles;
    const SlotDesc &D = a.sd[s];
    const TraceCtx &B = reinterpret_cast<const TraceCtx *>(a.tctx)[s];
    const int N = D.N, nseg = D.nseg;
    const int tw = D.tile_w, lw = __ffs(tw) - 1;
    const int i0 = (tile_id % D.tiles_x) * tw, j0 = (tile_id / D.tiles_x) * (kTileRays >> lw);
    const size_t px0 = (size_t)s * a.ray_stride, tile = (size_t)s * a.n_blocks_x + tile_id;
    WalkShared &S = s_walk[w];
    Cands cd;
    cd.n = 0;
    cd.id = reinterpret_cast<int *>(S.node) + lane;
    // ---- the first warp: primary hits
    float wgt = 1.0f;
    unsigned hitbits = 0u;
    bool clean = true, live = false, inside = false, seen = false;
    int nseg_done = 0, ray = 0;
    Best32 h;
    h.part = h.tl = -1;
    h.b1 = h.b2 = 0.0f;
    if (w == 0) {
        const int i = i0 + (lane & (tw - 1)), j = j0 + (lane >> lw);
        ray = i * N + j;
        inside = i < N && j < N;
        const bool skip_slot = B.skip != 0, bad = a.rast_bad[s] != 0;
        const unsigned long long pk = inside && !skip_slot ? __ldcs(a.pix_key + px0 + ray) : ~0ull;
        live = seen = inside && !skip_slot && (bad || pk != ~0ull);  // (all ones: no hit, no candidate)
        nseg_done = inside ? 1 : 0;
        const bool some = __any_sync(0xffffffffu, live);
        if (HITS && inside && B.skip != kSkipDist && !live) {
            int32_t *hq = a.hits + (px0 + ray) * a.seg_stride;
            for (int k = 0; k < nseg; k++) hq[k] = -1;
        }
        if (lane == 0) {
            F.n_list = some ? 0 : -1;
            F.flags = 0;
        }
        __syncwarp();  // (lanes add their flags below)
        if (!some) {
            const unsigned n = (unsigned)__popc(__ballot_sync(0xffffffffu, inside));
            if (lane == 0) a.amb_count[tile] = 0;
            if (!skip_slot) {
                if (lane < 6) a.partials[tile * 6 + lane] = 0.0f;
                if (lane < kCntRay) a.pcounts[tile * kCnt + lane] = lane == 1 ? n : 0u;  // (segments)
            }
        } else {
            for (int k = 0; k < 6; k++) F.acc[k][lane] = 0.0f;
            for (int k = 0; k < 3; k++) F.d[k][lane] = B.dir[k];
            F.res[lane] = -1;
        }
        if (live) {
            const float uc = fmaf((float)i + 0.5f, B.du32, B.umin32);
            const float vc = fmaf((float)j + 0.5f, B.dv32, B.vmin32);
            const unsigned pn = key_cands(pk);
            if (!bad && pix_listed(pn, slot_over(a, s))) {
                if (!key_none(pk)) {
                    // the raster's nearest certain hit; its barycentric weights as the traversal forms them
                    const unsigned id = (unsigned)pk & kKeyId;
                    h.part = (int)(id >> 24);
                    h.tl = (int)(id & 0xffffffu);
                    const PartView &pv = B.part[h.part];
                    // (read by the shading below; on their way meanwhile)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(pv.tri + (size_t)h.tl * 3));
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(B.grp + pv.tri_begin + h.tl));
                    const int4 vi = __ldg(pv.v4 + h.tl);
                    const Prim32 q = prim_core(__ldg(B.vview + vi.x), __ldg(B.vview + vi.y), __ldg(B.vview + vi.z), uc,
                                               vc, B.w0_32);
                    const float id32 = 1.0f / q.det;
                    h.b1 = q.V * id32;
                    h.b2 = q.W * id32;
                }
                cd.n = (int)pn;
                for (int c = 0; c < min((int)pn, kPixCand); c++) cd.id[c * kCandStride] = (int)a.pix_cand[(px0 + ray) * kPixCand + c];
                if (pn > (unsigned)kPixCand) cd.n = over_cands(slot_over(a, s), (unsigned)ray, (int)pn, cd.id);
            } else {
                // a traversed primary segment starts at its pixel on the window
                Ray32 r;
                for (int k = 0; k < 3; k++) {
                    r.d[k] = B.dir[k];
                    r.o[k] = fmaf((float)i + 0.5f, B.du[k], fmaf((float)j + 0.5f, B.dv[k], B.org[k]));
                }
                ray_setup(r);
                const Counts none = {0u, 0u, 0u, {0u, 0u, 0u, 0u}, 0};
                const Near32 o = nearest32_primary<false, false>(B, r, uc, vc, B.delta_p, B.tau_p, none, cd);
                h = o.b;
                cd.n = o.cand_n;
                clean = o.ok != 0;
                if (o.cn.flags) atomicOr(&F.flags, o.cn.flags);
            }
        }
        const bool want = live && clean && cd.n > 0;
        if (__any_sync(0xffffffffu, want))  // settle in FP64
            h = resolve64_warp(B, want, N, i, j, 0, &F.hpt[0][lane], kTileRays, -1, cd, h);
        live = live && clean && h.part >= 0;
    }
    float delta = B.delta_p, tau = 0.0f;
    for (int seg = 0;; seg++) {
        if (w == 0) {
            // shade the hits of segment seg and reflect
            if (live) {
                F.hpt[seg][lane] = (h.part << 24) | h.tl;
                hitbits |= 1u << seg;
                float acc[6], d[3];
                for (int k = 0; k < 6; k++) acc[k] = F.acc[k][lane];
                for (int k = 0; k < 3; k++) d[k] = F.d[k][lane];
                const Shade32 sh = shade_hit(B, h, d, wgt, acc);
                for (int k = 0; k < 6; k++) F.acc[k][lane] = acc[k];
                clean = !no_normal(sh);
                wgt *= sh.rs;
                live = clean && seg + 1 < nseg && wgt != 0.0f;
                if (live) {
                    Ray32 r;
                    for (int k = 0; k < 3; k++) {
                        r.o[k] = sh.hp[k];
                        r.d[k] = d[k] - 2.0f * sh.dn * sh.n[k];
                        F.d[k][lane] = r.d[k];
                    }
                    // the reflected ray leaves the hit triangle's plane at |dn|: its coplanar group can
                    // only be met within dev / |dn| of the origin, inside the self-hit distance eps
                    const int2 g = __ldg(B.grp + B.part[h.part].tri_begin + h.tl);
                    F.gskip[lane] = fabsf(sh.dn) * B.eps32 > 16.0f * __int_as_float(g.y) ? g.x : kNoGroup;
                    ray_setup(r);
                    F.ra[lane] = make_float4(r.o[0], r.o[1], r.o[2], __int_as_float(sh.orig));
                    F.rb[lane] = make_float4(r.inv[0], r.inv[1], r.inv[2], __int_as_float(h.part));
                    F.rc[lane] = make_float4(r.Sx, r.Sy, r.Sz, __int_as_float(r.code));
                    nseg_done++;
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, live);
            if (live) F.list[__popc(m & ((1u << lane) - 1u))] = lane;
            if (lane == 0 && F.n_list >= 0) F.n_list = __popc(m);
        }
        __syncthreads();
        const int n = F.n_list;
        if (n < 0) return;  // an empty tile
        if (n == 0) break;
        // the origin error grows with the previous segment's bound
        // (the same for every ray of the segment: the lanes test each other's rays)
        delta = B.delta_s + 2.0f * delta;
        tau = 64.0f * delta + 32.0f * kU * (B.R + B.L);
        // ---- every warp: the walks of its share, every kFewWarps-th ray
        if (w < n) {
            const int at = w + kFewWarps * lane;
            const bool mine = at < n;
            const int tl = mine ? F.list[at] : 0;
            Ray32 r;
            int skip = -1, gpart = -1, gskip = kNoGroup;
            if (mine) {
                const float4 A = F.ra[tl], I = F.rb[tl], C = F.rc[tl];
                r.o[0] = A.x; r.o[1] = A.y; r.o[2] = A.z;
                r.inv[0] = I.x; r.inv[1] = I.y; r.inv[2] = I.z;
                for (int k = 0; k < 3; k++) r.oi[k] = r.o[k] * r.inv[k];
                r.Sx = C.x; r.Sy = C.y; r.Sz = C.z;
                r.code = __float_as_int(C.w);
                skip = __float_as_int(A.w);
                gpart = __float_as_int(I.w);
                gskip = F.gskip[tl];
            }
            Best32 b;
            Counts cn = {0u, 0u, 0u, {0u, 0u, 0u, 0u}, 0};
            const bool ok = walk_warp<false>(B, S, D.mesh, mine, r, skip, gpart, gskip, delta, tau, b, cn, cd);
            const bool want = mine && ok && cd.n > 0;
            if (__any_sync(0xffffffffu, want))  // settle in FP64
                b = resolve64_warp(B, want, N, i0 + (tl & (tw - 1)), j0 + (tl >> lw), seg + 1, &F.hpt[0][tl], kTileRays,
                                   skip, cd, b);
            if (mine) {
                F.res[tl] = !ok ? -2 : (b.part < 0 ? -1 : (b.part << 24) | b.tl);
                F.b1[tl] = b.b1;
                F.b2[tl] = b.b2;
                if (cn.flags) atomicOr(&F.flags, cn.flags);
            }
        }
        __syncthreads();
        if (w == 0 && live) {
            const int res = F.res[lane];
            clean = res != -2;
            live = res >= 0;
            h.part = res >> 24;
            h.tl = res & 0xffffff;
            h.b1 = F.b1[lane];
            h.b2 = F.b2[lane];
        }
    }
    if (w != 0) return;
    // the tile's results as the trace block leaves them
    if (HITS && seen && clean) {
        int32_t *hq = a.hits + (px0 + ray) * a.seg_stride;
        for (int k = 0; k < nseg; k++) {
            int o = -1;
            if ((hitbits >> k) & 1u) {
                const int hk = F.hpt[k][lane];
                o = __float_as_int(__ldg(B.part[hk >> 24].tri + (size_t)(hk & 0xffffff) * 3).w);
            }
            hq[k] = o;
        }
    }
    float fac[6];
    for (int k = 0; k < 6; k++) fac[k] = clean ? F.acc[k][lane] : 0.0f;
    Counts cn = {0u, 0u, 0u, {0u, 0u, 0u, 0u}, 0};
    tile_results<false>(a, s, tile_id, ray, fac, clean ? 0u : 1u, clean ? (unsigned)nseg_done : 0u, clean ? hitbits : 0u, cn,
                        F.flags);
}

// ------------------------------------------------------------- work queue
// The raster's second pass and the trace of a launch's slots as one persistent
// kernel over a queue of work items, handed out in this order: the second pass
// over small triangles (slot-major, 128 triangles an item), over the listed
// chunks of large triangles (kTraceWarps chunks an item, a warp each), then the
// trace blocks (kTraceWarps tiles an item).  A trace item of slot s may start
// once every second-pass item of slot s has finished, which its block waits for
// on the slot's completion counters.  Items are handed out in order and
// second-pass items never wait, so the items a trace item waits for are held by
// running blocks and every wait ends; each is bounded all the same (device
// time): past the bound the block sets the slot's timeout flag and the queue's
// abort flag (later waits give up at once), writes an empty result for its
// tiles and goes on, and the call reports SRP_ERR_TIMEOUT.
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr unsigned long long kQueueWaitNs = 2000000000ull;  // 2 s of device time
constexpr unsigned long long kQueueTestWaitNs = 2000000ull; // 2 ms when a test makes the wait run out
constexpr int kQueueBatch = 4;  // consecutive items a block claims at once

// Slot of second-pass item it: the last slot whose first item is <= it.
__device__ __forceinline__ int slot_of_rast_item(const SlotDesc *sd, int S, unsigned it)
{
    int lo = 0, hi = S - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if ((unsigned)__ldg(&sd[mid].rast0) <= it) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Wait (thread 0 of a block) until slot s's second raster pass is complete; 1
// when it is, 0 when the wait gave up.
__device__ int queue_wait(const TraceArgs &a, int s)
{
    const unsigned *q = a.qstate + kQSlot + 3 * s;
    const unsigned need_small = (unsigned)((a.sd[s].mesh->n_tris + 127) / 128) + (a.wait_test ? 1u : 0u);
    const unsigned need_big = ld_acquire(q + 2);  // final: counted by the chunk listing, an earlier launch
    const unsigned long long limit = a.wait_test ? kQueueTestWaitNs : kQueueWaitNs;
    const unsigned long long t0 = global_ns();
    unsigned ns = 32;
    while (true) {
        if (ld_acquire(q) >= need_small && ld_acquire(q + 1) >= need_big) return 1;
        if (ld_acquire(a.qstate + kQAbort)) break;
        if (global_ns() - t0 > limit) {
            atomicExch(a.qstate + kQAbort, 1u);
            break;
        }
        __nanosleep(ns);
        if (ns < 1024) ns *= 2;
    }
    atomicOr(&a.pose[s].flags, kFlagTimeout);
    return 0;
}

// An empty result for trace block vb (its wait gave up): no force, no counts,
// no hand-offs.
__device__ void trace_block_empty(const TraceArgs &a, int vb)
{
    const int s = slot_of_block(a.sd, a.n_slots, vb);
    const SlotDesc &D = a.sd[s];
    const int tile_id = (vb - D.tile0) * kTraceWarps + (int)(threadIdx.x >> 5);
    if (tile_id >= D.tiles || (threadIdx.x & 31) != 0) return;
    const size_t tile = (size_t)s * a.n_blocks_x + tile_id;
    for (int k = 0; k < 6; k++) a.partials[tile * 6 + k] = 0.0f;
    for (int k = 0; k < kCnt; k++) a.pcounts[tile * kCnt + k] = 0u;
    a.amb_count[tile] = 0;
}

template <bool COUNT, bool HITS>
__global__ void __launch_bounds__(kTileRays * kTraceWarps, 32 / kTraceWarps) k_queue(TraceArgs a)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char s_dyn[];
    TraceCtx &B = *reinterpret_cast<TraceCtx *>(s_dyn);
    int *s_hpt = reinterpret_cast<int *>(s_dyn + trace_ctx_dyn_bytes(a.ctx_parts));
    __shared__ int s_cand[kCand * kLaneStride];
    __shared__ unsigned s_item;
    __shared__ int s_ok, s_ready;  // s_ready: a slot whose second pass this block has seen complete
    const unsigned lane = threadIdx.x & 31u;
    const unsigned n_small = (unsigned)a.n_small_items;
    const unsigned n_big_e = min(ld_acquire(a.big_count), (unsigned)a.big_cap);
    const unsigned n_big = (n_big_e + kTraceWarps - 1) / kTraceWarps;
    const unsigned total = n_small + n_big + (unsigned)a.n_tiles;
    if (threadIdx.x == 0) s_ready = -1;
    for (;;) {
        __syncthreads();  // every warp is done with the previous item and its shared state
        if (threadIdx.x == 0) s_item = atomicAdd(a.qstate + kQHead, (unsigned)kQueueBatch);
        __syncthreads();
        const unsigned it0 = s_item;
        if (it0 >= total) break;
        const unsigned it1 = min(it0 + (unsigned)kQueueBatch, total);
        for (unsigned it = it0; it < it1; it++) {
        if (it > it0) __syncthreads();
        if (it < n_small) {
            const int s = slot_of_rast_item(a.sd, a.n_slots, it);
            raster_tri<1>(a, s, (int)(it - (unsigned)a.sd[s].rast0) * 128 + (int)threadIdx.x);
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                atomicAdd(a.qstate + kQSlot + 3 * s, 1u);
            }
        } else if (it < n_small + n_big) {
            const unsigned e = (it - n_small) * kTraceWarps + (threadIdx.x >> 5);
            if (e < n_big_e) {
                const int s = raster_big_entry<1>(a, e, lane);
                __syncwarp();
                if (lane == 0 && s >= 0) {
                    __threadfence();
                    atomicAdd(a.qstate + kQSlot + 3 * s + 1, 1u);
                }
            }
        } else {
            const int vb = (int)(it - n_small - n_big);
            if (threadIdx.x == 0) {
                const int s = slot_of_block(a.sd, a.n_slots, vb);
                s_ok = s == s_ready ? 1 : queue_wait(a, s);
                if (s_ok) s_ready = s;
            }
            __syncthreads();
            if (s_ok) trace_block<COUNT, HITS, true>(a, vb, B, s_cand, s_hpt);
            else trace_block_empty(a, vb);
        }
        }
    }
}

// ------------------------------------------------------------- FP64 path
struct Ray64 {
    double o[3], d[3];
    double Sx, Sy, Sz;
    int kx, ky, kz;
};

__device__ void ray64_setup(Ray64 &r)
{
    double ax = fabs(r.d[0]), ay = fabs(r.d[1]), az = fabs(r.d[2]);
    int kz = (ax > ay) ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    int kx = kz == 2 ? 0 : kz + 1;
    int ky = kx == 2 ? 0 : kx + 1;
    double dz = pickd(r.d[0], r.d[1], r.d[2], kz);
    if (dz < 0.0) { int t = kx; kx = ky; ky = t; }
    r.kx = kx; r.ky = ky; r.kz = kz;
    const double rz = 1.0 / dz;
    r.Sx = pickd(r.d[0], r.d[1], r.d[2], kx) * rz;
    r.Sy = pickd(r.d[0], r.d[1], r.d[2], ky) * rz;
    r.Sz = rz;
}

__device__ void tri_v64(const TraceCtx &B, int p, int tl, double *v)
{
    const PartView &pv = B.part[p];
    int t = pv.tri_begin + tl;
    for (int c = 0; c < 3; c++) {
        int vi = B.tri_vidx[3 * t + c] - pv.vert_begin;
        for (int k = 0; k < 3; k++) v[3 * c + k] = pv.v64[3 * vi + k];
    }
}

// FP64 signs and comparisons by their bits (an FP64 comparison holds the FP64 pipe
// like an addition: 64 cycles a warp): x < 0 and x > 0 of a number that is not NaN,
// a > b where b is not negative.
__device__ __forceinline__ bool neg64(double x)
{
    return __double2hiint(x) < 0 && ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) != 0;
}
__device__ __forceinline__ bool pos64(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool above64(double a, double b) { return __double_as_longlong(a) > __double_as_longlong(b); }
// the edge functions have both signs: the line misses the triangle
__device__ __forceinline__ bool missed64(double U, double V, double W)
{
    return (neg64(U) || neg64(V) || neg64(W)) && (pos64(U) || pos64(V) || pos64(W));
}
__device__ __forceinline__ bool zero64(double x) { return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) == 0; }
// the nearer of two hits above tlo >= 0: equal distances go to the lowest original id
__device__ __forceinline__ bool nearer64(double t, int orig, double tlo, double bt, int bo)
{
    return above64(t, tlo) && (above64(bt, t) || (__double_as_longlong(t) == __double_as_longlong(bt) && orig < bo));
}

// FP64 watertight edge functions and scaled depth of triangle v against ray r.
__device__ __forceinline__ void wt64(const Ray64 &r, const double *v, double &U, double &V, double &W, double &det,
                                     double &T)
{
    double A[3], Bv[3], C[3];
    for (int k = 0; k < 3; k++) { A[k] = v[k] - r.o[k]; Bv[k] = v[3 + k] - r.o[k]; C[k] = v[6 + k] - r.o[k]; }
    double Akz = pickd(A[0], A[1], A[2], r.kz), Bkz = pickd(Bv[0], Bv[1], Bv[2], r.kz), Ckz = pickd(C[0], C[1], C[2], r.kz);
    double Ax = pickd(A[0], A[1], A[2], r.kx) - r.Sx * Akz, Ay = pickd(A[0], A[1], A[2], r.ky) - r.Sy * Akz;
    double Bx = pickd(Bv[0], Bv[1], Bv[2], r.kx) - r.Sx * Bkz, By = pickd(Bv[0], Bv[1], Bv[2], r.ky) - r.Sy * Bkz;
    double Cx = pickd(C[0], C[1], C[2], r.kx) - r.Sx * Ckz, Cy = pickd(C[0], C[1], C[2], r.ky) - r.Sy * Ckz;
    U = __dsub_rn(__dmul_rn(Cx, By), __dmul_rn(Cy, Bx));
    V = __dsub_rn(__dmul_rn(Ax, Cy), __dmul_rn(Ay, Cx));
    W = __dsub_rn(__dmul_rn(Bx, Ay), __dmul_rn(By, Ax));
    det = U + V + W;
    T = U * (r.Sz * Akz) + V * (r.Sz * Bkz) + W * (r.Sz * Ckz);
}

// The exact (FP64) ray of segment seg > 0: from the pixel centre through the planes of the earlier segments' hits.
__device__ __forceinline__ void segment_ray64(const TraceCtx &B, double uc, double vc, double w0, int seg, const int *hpt,
                                              int hps, Ray64 &r)
{
    for (int k = 0; k < 3; k++) { r.o[k] = uc * B.u[k] + vc * B.v[k] + w0 * B.d[k]; r.d[k] = B.d[k]; }
    double v[9];
    for (int s = 0; s < seg; s++) {
        // hit point on the plane of the segment's triangle, then the specular direction
        const int hs = hpt[s * hps];
        tri_v64(B, hs >> 24, hs & 0xffffff, v);
        double e1[3], e2[3], m[3], ao[3];
        for (int k = 0; k < 3; k++) { e1[k] = v[3 + k] - v[k]; e2[k] = v[6 + k] - v[k]; ao[k] = v[k] - r.o[k]; }
        m[0] = e1[1] * e2[2] - e1[2] * e2[1];
        m[1] = e1[2] * e2[0] - e1[0] * e2[2];
        m[2] = e1[0] * e2[1] - e1[1] * e2[0];
        double dm = r.d[0] * m[0] + r.d[1] * m[1] + r.d[2] * m[2];
        double t = (ao[0] * m[0] + ao[1] * m[1] + ao[2] * m[2]) / dm;
        double f = 2.0 * dm / (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
        for (int k = 0; k < 3; k++) { r.o[k] = r.o[k] + t * r.d[k]; r.d[k] = r.d[k] - f * m[k]; }
    }
    ray64_setup(r);

}

// The FP64 test of a primary segment, in the view frame: edge functions and scaled depth of triangle tl.
__device__ __forceinline__ void prim64(const TraceCtx &B, const PartView &pv, int tl, double uc, double vc, double w0,
                                       double &U, double &V, double &W, double &det, double &T)
{
    int4 vi = __ldg(pv.v4 + tl);
    const double *a = B.vview64 + 3 * (size_t)vi.x, *b = B.vview64 + 3 * (size_t)vi.y,
                 *q = B.vview64 + 3 * (size_t)vi.z;
    double Ax = a[0] - uc, Ay = a[1] - vc, Bx = b[0] - uc, By = b[1] - vc, Cx = q[0] - uc, Cy = q[1] - vc;
    U = __dsub_rn(__dmul_rn(Cx, By), __dmul_rn(Cy, Bx));
    V = __dsub_rn(__dmul_rn(Ax, Cy), __dmul_rn(Ay, Cx));
    W = __dsub_rn(__dmul_rn(Bx, Ay), __dmul_rn(By, Ax));
    det = U + V + W;
    T = U * (a[2] - w0) + V * (b[2] - w0) + W * (q[2] - w0);
}

// Settle one segment's uncertain FP32 decisions in FP64: the FP64 test of each
// candidate and of the nearest certain FP32 hit against the segment's exact
// ray; the nearest t above the self-hit threshold wins, equal t goes to the
// lowest original triangle id (the rule of the FP64 re-trace).  Every other
// triangle was certainly missed, certainly farther, or culled beyond the
// certain hit plus its band.  Primary segments are tested in the view frame
// (the ray is the line through the FP64 pixel centre along d; vertex
// projections computed once per evaluation in FP64); a specular segment's ray
// is the FP64 chain through the earlier segments' hit triangles, tested with
// the FP64 watertight test.  FP64 is slow on this GPU: no square roots, one
// division per candidate, barycentric weights for the winner only.
// hpt: the ray's column of the block's hit records (segment s at hpt[s * hps]).
__device__ __noinline__ Best32 resolve64(const TraceCtx &B, int N, int i, int j, int seg, const int *hpt, int hps,
                                         int skip, Cands cd, Best32 best)
{
    double bt = INFINITY, bU = 0.0, bV = 0.0, bW = 0.0;
    int bp = -1, btl = -1, bo = 0x7fffffff;
    const double uc = B.umin + pix64(((double)i + 0.5) * B.Du, B.rN, N);
    const double vc = B.vmin + pix64(((double)j + 0.5) * B.Dv, B.rN, N);
    const double w0 = B.wmin - kStandoff;
    Ray64 r;
    double tlo = 0.0;
    if (seg > 0) {
        segment_ray64(B, uc, vc, w0, seg, hpt, hps, r);
        tlo = B.eps;
    }
    for (int c = 0; c <= cd.n; c++) {
        int p, tl;
        if (c < cd.n) { const int id = cd.id[c * kCandStride]; p = id >> 24; tl = id & 0xffffff; }
        else if (best.part >= 0) { p = best.part; tl = best.tl; }
        else break;
        const PartView &pv = B.part[p];
        int orig = __float_as_int(__ldg(pv.tri + (size_t)tl * 3).w);
        if (orig == skip) continue;
        double U, V, W, det, T;
        if (seg == 0) {
            prim64(B, pv, tl, uc, vc, w0, U, V, W, det, T);
        } else {
            double v[9];
            tri_v64(B, p, tl, v);
            wt64(r, v, U, V, W, det, T);
        }
        if (missed64(U, V, W) || zero64(det)) continue;
        double t = T / det;
        if (nearer64(t, orig, tlo, bt, bo)) {
            bt = t; bp = p; btl = tl; bo = orig; bU = det; bV = V; bW = W;
        }
    }
    best.t = (float)bt;
    best.part = bp;
    best.tl = btl;
    best.b1 = bp >= 0 ? (float)(bV / bU) : 0.f;
    best.b2 = bp >= 0 ? (float)(bW / bU) : 0.f;
    return best;
}

// resolve64 by a warp (every lane calls it; `want` where the lane's ray has candidates): the
// (ray, triangle) pairs are dealt to the lanes, so a step of FP64 tests covers up to 32 of
// them.  An FP64 instruction takes the warp 64 cycles for one lane or for all: a ray with
// three triangles to test costs 150 of them instead of 270.  The same decisions, by the same tests.
__device__ __noinline__ Best32 resolve64_warp(const TraceCtx &B, bool want, int N, int i, int j, int seg, const int *hpt,
                                              int hps, int skip, Cands cd, Best32 best)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    __syncwarp();  // the lanes read each other's candidate columns below; votes and shuffles order no memory
    const double uc = B.umin + pix64(((double)i + 0.5) * B.Du, B.rN, N);
    const double vc = B.vmin + pix64(((double)j + 0.5) * B.Dv, B.rN, N);
    const double w0 = B.wmin - kStandoff, tlo = seg > 0 ? B.eps : 0.0;
    Ray64 r;
    r.o[0] = uc; r.o[1] = vc; r.o[2] = 0.0;
    r.Sx = r.Sy = r.Sz = 0.0;
    r.kx = r.ky = r.kz = 0;
    if (seg > 0 && want) segment_ray64(B, uc, vc, w0, seg, hpt, hps, r);
    // the lane's pairs: its candidates, then its nearest certain hit
    const int mine = want ? cd.n + (best.part >= 0 ? 1 : 0) : 0;
    int end = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(kAll, end, o);
        if (lane >= o) end += x;
    }
    const int first = end - mine, total = __shfl_sync(kAll, end, 31), most = __reduce_max_sync(kAll, mine);
    const int kk = r.kx | r.ky << 2 | r.kz << 4;
    const int hit = best.part >= 0 ? (best.part << 24) | best.tl : 0;
    double bt = INFINITY, bU = 1.0, bV = 0.0, bW = 0.0;
    int bid = -1, bo = 0x7fffffff;
    for (int p0 = 0; p0 < total; p0 += 32) {
        const int p = min(p0 + lane, total - 1);
        int src = 0;  // the lane whose pair it is: the first with end > p
        for (int h = 16; h; h >>= 1)
            if (__shfl_sync(kAll, end, src + h - 1) <= p) src += h;
        const int c = p - __shfl_sync(kAll, first, src), cn = __shfl_sync(kAll, cd.n, src);
        const unsigned long long col = __shfl_sync(kAll, reinterpret_cast<unsigned long long>(cd.id), src);
        const int sh = __shfl_sync(kAll, hit, src), sk = __shfl_sync(kAll, skip, src), k = __shfl_sync(kAll, kk, src);
        Ray64 q;
        for (int x = 0; x < 3; x++) q.o[x] = __shfl_sync(kAll, r.o[x], src);
        q.Sx = __shfl_sync(kAll, r.Sx, src); q.Sy = __shfl_sync(kAll, r.Sy, src); q.Sz = __shfl_sync(kAll, r.Sz, src);
        q.kx = k & 3; q.ky = (k >> 2) & 3; q.kz = k >> 4;
        const int id = c < cn ? reinterpret_cast<const int *>(col)[c * kCandStride] : sh;
        const PartView &pv = B.part[id >> 24];
        const int tl = id & 0xffffff;
        int orig = __float_as_int(__ldg(pv.tri + (size_t)tl * 3).w);
        double U, V, W, det, T, t = INFINITY;
        if (seg == 0) {
            prim64(B, pv, tl, q.o[0], q.o[1], w0, U, V, W, det, T);
        } else {
            double v[9];
            tri_v64(B, id >> 24, tl, v);
            wt64(q, v, U, V, W, det, T);
        }
        if (orig == sk || missed64(U, V, W) || zero64(det)) orig = -1;
        else t = T / det;
        // each ray's nearest, in its lane
        int win = -1;
        for (int e = 0; e < most; e++) {
            const int l = first + e - p0;
            const bool own = e < mine && l >= 0 && l < 32;
            const double te = __shfl_sync(kAll, t, l & 31);
            const int oe = __shfl_sync(kAll, orig, l & 31);
            if (own && oe >= 0 && nearer64(te, oe, tlo, bt, bo)) { bt = te; bo = oe; win = l; }
        }
        const double wU = __shfl_sync(kAll, det, win & 31), wV = __shfl_sync(kAll, V, win & 31),
                     wW = __shfl_sync(kAll, W, win & 31);
        const int wi = __shfl_sync(kAll, id, win & 31);
        if (win >= 0) { bU = wU; bV = wV; bW = wW; bid = wi; }
    }
    if (want) {
        best.t = (float)bt;
        best.part = bid < 0 ? -1 : bid >> 24;
        best.tl = bid < 0 ? -1 : bid & 0xffffff;
        best.b1 = bid >= 0 ? (float)(bV / bU) : 0.f;
        best.b2 = bid >= 0 ? (float)(bW / bU) : 0.f;
    }
    return best;
}

// True when the FP32 world-frame test shows the triangle certainly misses the
// ray: some edge function certainly negative and another certainly positive,
// with the per-triangle error bound of the secondary-ray test.
__device__ __forceinline__ bool outside32(const Ray32 &r, float4 a, float4 b, float4 c, float delta)
{
    const float u4 = 4.0f * kU;
    float A0 = a.x - r.o[0], A1 = a.y - r.o[1], A2 = a.z - r.o[2];
    float B0 = b.x - r.o[0], B1 = b.y - r.o[1], B2 = b.z - r.o[2];
    float C0 = c.x - r.o[0], C1 = c.y - r.o[1], C2 = c.z - r.o[2];
    float Akz = pick(A0, A1, A2, r.kz()), Bkz = pick(B0, B1, B2, r.kz()), Ckz = pick(C0, C1, C2, r.kz());
    float Ax = fmaf(-r.Sx, Akz, pick(A0, A1, A2, r.kx())), Ay = fmaf(-r.Sy, Akz, pick(A0, A1, A2, r.ky()));
    float Bx = fmaf(-r.Sx, Bkz, pick(B0, B1, B2, r.kx())), By = fmaf(-r.Sy, Bkz, pick(B0, B1, B2, r.ky()));
    float Cx = fmaf(-r.Sx, Ckz, pick(C0, C1, C2, r.kx())), Cy = fmaf(-r.Sy, Ckz, pick(C0, C1, C2, r.ky()));
    float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    float dz = fmaxf(fmaxf(fabsf(Akz), fabsf(Bkz)), fabsf(Ckz)) + fmaxf(fmaxf(fabsf(Ax), fabsf(Bx)), fabsf(Cx)) +
               fmaxf(fmaxf(fabsf(Ay), fabsf(By)), fabsf(Cy));
    float dc = fmaf(16.0f * kU, dz, delta);
    float eU = dc * (fabsf(Bx) + fabsf(By) + fabsf(Cx) + fabsf(Cy)) + u4 * (fabsf(Cx * By) + fabsf(Cy * Bx));
    float eV = dc * (fabsf(Ax) + fabsf(Ay) + fabsf(Cx) + fabsf(Cy)) + u4 * (fabsf(Ax * Cy) + fabsf(Ay * Cx));
    float eW = dc * (fabsf(Ax) + fabsf(Ay) + fabsf(Bx) + fabsf(By)) + u4 * (fabsf(Bx * Ay) + fabsf(By * Ax));
    bool neg = (U < -eU) || (V < -eV) || (W < -eW);
    bool pos = (U > eU) || (V > eV) || (W > eW);
    return neg && pos;
}

// Nearest hit in FP64 (same BVH; boxes tested with the rounded ray, whose
// deviation from the FP64 ray is far below the box padding).
__device__ void nearest64(const TraceCtx &B, const Ray64 &r, double tlo, int skip, double &bt, int &bpart, int &btl,
                          int &borig, int &flags)
{
    bt = INFINITY;
    bpart = -1; btl = -1; borig = 0x7fffffff;
    Ray32 q;
    for (int k = 0; k < 3; k++) { q.o[k] = (float)r.o[k]; q.d[k] = (float)r.d[k]; }
    ray_setup(q);
    const float slack = 4.0f * B.pad;
    // bound on the coordinate error of the rounded ray and FP32 vertices, for the
    // FP32 pre-test that skips triangles the ray certainly misses
    float omax = fmaxf(fmaxf(fabsf(q.o[0]), fabsf(q.o[1])), fabsf(q.o[2]));
    const float dq = 2.0f * kU * (omax + B.R);
    int stack[kStack];
    for (int p = 0; p < B.n_parts; p++) {
        const PartView &pv = B.part[p];
        float thi = (float)bt + slack;
        if (box_enter(pv.box[0], pv.box[3], pv.box[1], pv.box[4], pv.box[2], pv.box[5], q.inv, q.oi,
                      (float)tlo - slack, thi) == INFINITY)
            continue;
        int sp = 0, ref = pv.root, iters = 0;
        while (true) {
            if (++iters > pv.limit) { flags |= kFlagStack; break; }
            if (ref >= 0) {
                const int n = node4_step(pv.node + (size_t)ref * kNode4, q.inv, q.oi, q.code, (float)tlo - slack,
                                         (float)bt + slack, ref, stack, sp);
                if (n < 0) { flags |= kFlagStack; break; }
                if (n > 0) continue;
            } else {
                int tl = ~ref;
                const float4 *tr = pv.tri + (size_t)tl * 3;
                float4 fa = __ldg(tr), fb = __ldg(tr + 1), fc = __ldg(tr + 2);
                int orig = __float_as_int(fa.w);
                if (orig != skip && !outside32(q, fa, fb, fc, dq)) {
                    double v[9];
                    tri_v64(B, p, tl, v);
                    double U, V, W, det, T;
                    wt64(r, v, U, V, W, det, T);
                    if (!missed64(U, V, W) && !zero64(det)) {
                        const double t = T / det;
                        if (nearer64(t, orig, tlo, bt, borig)) { bt = t; bpart = p; btl = tl; borig = orig; }
                    }
                }
            }
            if (sp == 0) break;
            ref = stack[--sp];
        }
    }
}

// nearest64 of one ray by a warp (every lane calls it with the same ray): lanes take
// the nodes and triangles of one list, so a step's loads and a triangle's FP64 test
// cover up to 32 of them.  The result is the same: the least (t, original id) of the
// triangles not certainly missed or beyond it, in whatever order they are met.
constexpr int kWalk64 = 64;  // list entries (part, reference) beside the depth-first reserve
struct Walk64 {
    int2 e[kWalk64 + kStack];
};
__device__ __noinline__ void nearest64_warp(const TraceCtx &B, Walk64 &S, const Ray64 &r, double tlo, int skip,
                                            double &bt, int &bpart, int &btl, int &borig, int &flags)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    bt = INFINITY;
    bpart = -1; btl = -1; borig = 0x7fffffff;
    Ray32 q;
    for (int k = 0; k < 3; k++) { q.o[k] = (float)r.o[k]; q.d[k] = (float)r.d[k]; }
    ray_setup(q);
    const float slack = 4.0f * B.pad, tn = (float)tlo - slack;
    const float omax = fmaxf(fmaxf(fabsf(q.o[0]), fabsf(q.o[1])), fabsf(q.o[2]));
    const float dq = 2.0f * kU * (omax + B.R);
    // the parts whose box the ray enters, a lane each
    int n, limit;
    {
        bool in = false;
        int lim = 0;
        if (lane < B.n_parts) {
            const PartView &pv = B.part[lane];
            in = box_enter(pv.box[0], pv.box[3], pv.box[1], pv.box[4], pv.box[2], pv.box[5], q.inv, q.oi, tn, INFINITY) !=
                 INFINITY;
            lim = in ? pv.limit : 0;
        }
        const unsigned m = __ballot_sync(kAll, in);
        if (in) S.e[__popc(m & below)] = make_int2(lane, B.part[lane].root);
        n = __popc(m);
        limit = __reduce_add_sync(kAll, lim);
    }
    __syncwarp();
    while (n > 0) {
        // as many as their children have room for; one at a time at the end of the room,
        // which is then a depth-first walk and stays within the reserve
        const int m = min(min(n, 32), max(1, (kWalk64 - n) / 3));
        if ((limit -= m) < 0) { flags |= kFlagStack; break; }
        const bool mine = lane < m;
        int2 e = make_int2(0, 0);
        if (mine) e = S.e[n - 1 - lane];
        n -= m;
        __syncwarp();
        int4 c = make_int4(0, 0, 0, 0);
        bool in[4] = {false, false, false, false};
        bool test = false;
        int orig = 0x7fffffff;
        const float thi = (float)bt + slack;
        if (mine && e.y >= 0) {
            const float4 *nd = B.part[e.x].node + (size_t)e.y * kNode4;
            const int ox = q.code & 1, oy = (q.code >> 1) & 1, oz = (q.code >> 2) & 1;
            const float4 nx = __ldg(nd + ox), fx = __ldg(nd + 1 - ox), ny = __ldg(nd + 2 + oy), fy = __ldg(nd + 3 - oy),
                         nz = __ldg(nd + 4 + oz), fz = __ldg(nd + 5 - oz);
            c = __ldg(reinterpret_cast<const int4 *>(nd + 6));
            in[0] = box_enter_nf(nx.x, fx.x, ny.x, fy.x, nz.x, fz.x, q.inv, q.oi, tn, thi) != INFINITY;
            in[1] = box_enter_nf(nx.y, fx.y, ny.y, fy.y, nz.y, fz.y, q.inv, q.oi, tn, thi) != INFINITY;
            in[2] = box_enter_nf(nx.z, fx.z, ny.z, fy.z, nz.z, fz.z, q.inv, q.oi, tn, thi) != INFINITY;
            in[3] = box_enter_nf(nx.w, fx.w, ny.w, fy.w, nz.w, fz.w, q.inv, q.oi, tn, thi) != INFINITY;
        } else if (mine) {
            const float4 *tr = B.part[e.x].tri + (size_t)(~e.y) * 3;
            const float4 fa = __ldg(tr), fb = __ldg(tr + 1), fc = __ldg(tr + 2);
            orig = __float_as_int(fa.w);
            test = orig != skip && !outside32(q, fa, fb, fc, dq);
        }
        const int ck[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const unsigned mk = __ballot_sync(kAll, in[k]);
            if (in[k]) S.e[n + __popc(mk & below)] = make_int2(e.x, ck[k]);
            n += __popc(mk);
        }
        if (__any_sync(kAll, test)) {
            double t = INFINITY;
            bool hit = false;
            if (test) {
                double v[9], U, V, W, det, T;
                tri_v64(B, e.x, ~e.y, v);
                wt64(r, v, U, V, W, det, T);
                if (!missed64(U, V, W) && !zero64(det)) {
                    t = T / det;
                    hit = nearer64(t, orig, tlo, bt, borig);
                }
            }
            unsigned todo = __ballot_sync(kAll, hit);
            while (todo) {  // (few: hits nearer than what the earlier steps left)
                const int l = __ffs(todo) - 1;
                todo &= todo - 1u;
                const double tl = __shfl_sync(kAll, t, l);
                const int ol = __shfl_sync(kAll, orig, l), pl = __shfl_sync(kAll, e.x, l), rl = __shfl_sync(kAll, e.y, l);
                if (nearer64(tl, ol, tlo, bt, borig)) { bt = tl; bpart = pl; btl = ~rl; borig = ol; }
            }
        }
        __syncwarp();
    }
}

// Re-trace of one handed-off ray, FP64 from the pixel definition; adds to acc.
// (walk: by the whole warp, every lane with the same ray; null: by one lane)
__device__ __noinline__ void refine_ray(const TraceCtx &B, const TraceArgs &a, int s, int ray, Walk64 *walk, double *acc,
                                        int &flags)
{
    const int N = a.sd[s].N, nseg = a.sd[s].nseg;
    int i = ray / N, j = ray % N;
    Ray64 r;
    double uc = B.umin + pix64(((double)i + 0.5) * B.Du, B.rN, N);
    double vc = B.vmin + pix64(((double)j + 0.5) * B.Dv, B.rN, N);
    double w0 = B.wmin - kStandoff;
    for (int k = 0; k < 3; k++) { r.o[k] = uc * B.u[k] + vc * B.v[k] + w0 * B.d[k]; r.d[k] = B.d[k]; }
    double wgt = 1.0;
    int skip = -1, nseg_done = 0;
    int32_t *hp = a.hits ? a.hits + ((size_t)s * a.ray_stride + ray) * a.seg_stride : nullptr;
    if (hp) for (int k = 0; k < nseg; k++) hp[k] = -1;
    for (int seg = 0; seg < nseg; seg++) {
        ray64_setup(r);
        double t;
        int hpart, htl, horig;
        nseg_done++;
        if (walk) nearest64_warp(B, *walk, r, seg == 0 ? 0.0 : B.eps, skip, t, hpart, htl, horig, flags);
        else nearest64(B, r, seg == 0 ? 0.0 : B.eps, skip, t, hpart, htl, horig, flags);
        if (hpart < 0) break;
        if (hp) hp[seg] = horig;
        acc[8 + seg] += 1.0;
        double v[9];
        tri_v64(B, hpart, htl, v);
        double e1[3], e2[3], n[3];
        for (int k = 0; k < 3; k++) { e1[k] = v[3 + k] - v[k]; e2[k] = v[6 + k] - v[k]; }
        n[0] = e1[1] * e2[2] - e1[2] * e2[1];
        n[1] = e1[2] * e2[0] - e1[0] * e2[2];
        n[2] = e1[0] * e2[1] - e1[1] * e2[0];
        double nl = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
        for (int k = 0; k < 3; k++) n[k] /= nl;
        double dn = r.d[0] * n[0] + r.d[1] * n[1] + r.d[2] * n[2];
        int side = dn < 0.0 ? 0 : 1;
        double sg = side ? -1.0 : 1.0;
        unsigned mt = B.tri_mat[B.part[hpart].tri_begin + htl];
        int mi = side ? (int)(mt >> 16) : (int)(mt & 0xffffu);
        double rs = B.mat64[2 * mi], rd = B.mat64[2 * mi + 1];
        double c = -sg * dn;
        double F[3], x[3];
        for (int k = 0; k < 3; k++) F[k] = wgt * ((1.0 - rs) * r.d[k] - 2.0 * (rs * c + rd / 3.0) * sg * n[k]);
        for (int k = 0; k < 3; k++) x[k] = r.o[k] + t * r.d[k];
        double arm[3] = {x[0] - B.c_ref[0], x[1] - B.c_ref[1], x[2] - B.c_ref[2]};
        acc[0] += F[0]; acc[1] += F[1]; acc[2] += F[2];
        acc[3] += arm[1] * F[2] - arm[2] * F[1];
        acc[4] += arm[2] * F[0] - arm[0] * F[2];
        acc[5] += arm[0] * F[1] - arm[1] * F[0];
        wgt *= rs;
        if (seg + 1 >= nseg || wgt == 0.0) break;
        for (int k = 0; k < 3; k++) { r.d[k] = r.d[k] - 2.0 * dn * n[k]; r.o[k] = x[k]; }
        skip = horig;
    }
    acc[6] += 1.0;
    acc[7] += (double)nseg_done;
}

// ------------------------------------------------------- diffuse rays
// SplitMix64 output number c of the stream seeded with `seed` (Steele, Lea &
// Flood, OOPSLA 2014): the state after c + 1 golden-ratio increments, mixed.
__device__ __forceinline__ unsigned long long splitmix64_at(unsigned long long seed, unsigned long long c)
{
    unsigned long long z = seed + (c + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Cosine-weighted direction about the unit normal nf for sample counter c:
// uniforms from outputs 2c and 2c + 1 (top 53 bits), a uniform point of the
// unit disc lifted to the hemisphere (Malley's method), in the orthonormal
// basis of Duff et al. (JCGT 2017) around nf.
__device__ __forceinline__ void diffuse_dir(unsigned long long seed, unsigned long long c, const double *nf, double *w)
{
    const double u1 = (double)(splitmix64_at(seed, 2ull * c) >> 11) * 0x1.0p-53;
    const double u2 = (double)(splitmix64_at(seed, 2ull * c + 1ull) >> 11) * 0x1.0p-53;
    double sp, cp;
    sincospi(2.0 * u2, &sp, &cp);  // the angle 2 pi u2, reduced exactly (2 u2 is exact)
    const double rr = sqrt(u1), lz = sqrt(1.0 - u1);
    const double sign = copysign(1.0, nf[2]);
    const double a = -1.0 / (sign + nf[2]);
    const double b = nf[0] * nf[1] * a;
    const double t1[3] = {1.0 + sign * nf[0] * nf[0] * a, sign * b, -sign * nf[0]};
    const double t2[3] = {b, sign + nf[1] * nf[1] * a, -nf[1]};
    for (int k = 0; k < 3; k++) w[k] = rr * cp * t1[k] + rr * sp * t2[k] + lz * nf[k];
}

// Unit normal of a triangle from its FP64 vertices (v0 v1 v2 row-major).
__device__ __forceinline__ void tri_normal64(const double *v, double *n)
{
    double e1[3] = {v[3] - v[0], v[4] - v[1], v[5] - v[2]}, e2[3] = {v[6] - v[0], v[7] - v[1], v[8] - v[2]};
    n[0] = e1[1] * e2[2] - e1[2] * e2[1];
    n[1] = e1[2] * e2[0] - e1[0] * e2[2];
    n[2] = e1[0] * e2[1] - e1[1] * e2[0];
    const double il = 1.0 / sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    for (int k = 0; k < 3; k++) n[k] *= il;
}

// Settle an FP32 traversal's result in FP64: the FP64 watertight test of each
// uncertain candidate and of the nearest certain FP32 hit against the exact
// ray; the nearest t above tlo wins, equal t to the lowest original id.  Every
// other triangle was certainly missed, certainly farther, or culled beyond
// the certain hit plus its band.
__device__ void settle64(const TraceCtx &B, const Ray64 &r, double tlo, int skip, const Cands &cd, const Best32 &best,
                         double &bt, int &bp, int &btl)
{
    bt = INFINITY;
    bp = -1;
    btl = -1;
    int bo = 0x7fffffff;
    for (int c = 0; c <= cd.n; c++) {
        int p, tl;
        if (c < cd.n) { const int id = cd.id[c * kCandStride]; p = id >> 24; tl = id & 0xffffff; }
        else if (best.part >= 0) { p = best.part; tl = best.tl; }
        else break;
        const int orig = __float_as_int(__ldg(B.part[p].tri + (size_t)tl * 3).w);
        if (orig == skip) continue;
        double v[9], U, V, W, det, T;
        tri_v64(B, p, tl, v);
        wt64(r, v, U, V, W, det, T);
        if (missed64(U, V, W) || zero64(det)) continue;
        const double t = T / det;
        if (nearer64(t, orig, tlo, bt, bo)) { bt = t; bp = p; btl = tl; bo = orig; }
    }
}

// One diffuse sample a lane (`live` where it has one; every lane of the warp
// calls it) of counter c leaving hit point x of triangle `src` about the lit
// side's normal nf with weight wd: traced in FP32 with error-bounded
// decisions (as a secondary segment of the trace, the origin error being the
// rounding of the FP64 point), the uncertain ones settled in FP64; the FP64
// traversal when the candidate list overflows.  Its per-hit force and torque
// about c_ref are added to acc.
__device__ __forceinline__ void diffuse_sample(const TraceCtx &B, WalkShared &S, const MeshDev *mesh, bool live,
                                               unsigned long long seed, unsigned long long c, const double *x,
                                               const double *nf, int src, double wd, double *acc, int &flags)
{
    Ray64 r;
    double t = 0.0;
    int p = -1, tl = -1;
    {
        Ray32 q;
        if (live) {
            diffuse_dir(seed, c, nf, r.d);
            for (int e = 0; e < 3; e++) r.o[e] = x[e];
            ray64_setup(r);
            for (int e = 0; e < 3; e++) { q.o[e] = (float)r.o[e]; q.d[e] = (float)r.d[e]; }
            ray_setup(q);
        }
        const float delta = 2.0f * B.delta_s;
        const float tau = 64.0f * delta + 32.0f * kU * (B.R + B.L);
        Best32 b;
        Counts cn = {0u, 0u, 0u, {0u, 0u, 0u, 0u}, 0};
        Cands cd;
        cd.n = 0;
        cd.id = reinterpret_cast<int *>(S.node) + (threadIdx.x & 31);
        const bool ok = walk_warp<false>(B, S, mesh, live, q, src, -1, kNoGroup, delta, tau, b, cn, cd);
        if (!live) return;
        if (ok) {
            if (cd.n == 0) {
                // every FP32 decision was certain: the FP32 nearest hit is the FP64 one,
                // and its FP32 distance places the hit point for the torque arm
                p = b.part;
                tl = b.tl;
                t = (double)b.t;
            } else {
                settle64(B, r, B.eps, src, cd, b, t, p, tl);
            }
        } else {
            int orig;
            nearest64(B, r, B.eps, src, t, p, tl, orig, flags);
        }
        flags |= cn.flags;  // a walk bound is an error, as in the trace
    }
    if (p < 0) return;
    double v[9], n[3];
    tri_v64(B, p, tl, v);
    tri_normal64(v, n);
    const double dn = r.d[0] * n[0] + r.d[1] * n[1] + r.d[2] * n[2];
    const int side = dn < 0.0 ? 0 : 1;
    const double sg = side ? -1.0 : 1.0;
    const unsigned mt = B.tri_mat[B.part[p].tri_begin + tl];
    const int mi = side ? (int)(mt >> 16) : (int)(mt & 0xffffu);
    const double rs = B.mat64[2 * mi], rd = B.mat64[2 * mi + 1];
    const double cs = -sg * dn;
    double F[3], arm[3];
    for (int e = 0; e < 3; e++) {
        F[e] = wd * ((1.0 - rs) * r.d[e] - 2.0 * (rs * cs + rd / 3.0) * sg * n[e]);
        arm[e] = x[e] + t * r.d[e] - B.c_ref[e];
    }
    acc[0] += F[0]; acc[1] += F[1]; acc[2] += F[2];
    acc[3] += arm[1] * F[2] - arm[2] * F[1];
    acc[4] += arm[2] * F[0] - arm[0] * F[2];
    acc[5] += arm[0] * F[1] - arm[1] * F[0];
}

// Diffuse secondary rays of slot s, in three launches of kDiffBlocks blocks (k_dscan:
// one) a slot: the hits that emit (segments with a next level), their number, and K rays
// a hit of weight w rho_d / K, cosine-distributed about the lit side's normal, which
// deposit the per-hit law at theirs.  Sums per block in a fixed order: the result is
// reproducible.
// Step 1: a thread per primary ray replays its specular chain in
// FP64 through the recorded hit triangles and writes one record per hit that
// emits (a segment with a next level, rho_d > 0) to the ray's slots of the
// dense array, and the number of records.
__global__ void __launch_bounds__(kLaneStride) k_demit(TraceArgs a)
{
    pdl_enter();
    __shared__ TraceCtx B;
    const int s = blockIdx.y;
    if ((size_t)blockIdx.x * blockDim.x >= (size_t)a.sd[s].N * a.sd[s].N) return;  // no rays (uniform)
    load_ctx(B, a, s);
    __syncthreads();
    const SlotDesc &D = a.sd[s];
    const int N = D.N, nseg = D.nseg, K = a.n_diffuse;
    const size_t R = (size_t)N * N;
    int *cnt = a.dcnt + (size_t)s * a.ray_stride;
    for (size_t ray = (size_t)blockIdx.x * blockDim.x + threadIdx.x; ray < R; ray += (size_t)gridDim.x * blockDim.x) {
        int ne = 0;
        if (!B.skip) {
            const int *tri_pos = D.mesh->tri_pos;
            const int32_t *hq = a.hits + ((size_t)s * a.ray_stride + ray) * a.seg_stride;
            DEmit *out = a.demit + ((size_t)s * a.ray_stride + ray) * (size_t)(nseg - 1);
            const int i = (int)(ray / N), j = (int)(ray % N);
            const double uc = B.umin + pix64(((double)i + 0.5) * B.Du, B.rN, N);
            const double vc = B.vmin + pix64(((double)j + 0.5) * B.Dv, B.rN, N);
            const double w0 = B.wmin - kStandoff;
            double o[3], d[3];
            for (int k = 0; k < 3; k++) { o[k] = uc * B.u[k] + vc * B.v[k] + w0 * B.d[k]; d[k] = B.d[k]; }
            double wgt = 1.0;
            for (int k = 0; k + 1 < nseg; k++) {
                const int h = hq[k];
                if (h < 0) break;
                const int t = __ldg(tri_pos + h);
                const int p = part_of_sorted(D.mesh, t);
                const int tl = t - B.part[p].tri_begin;
                double v[9], n[3];
                tri_v64(B, p, tl, v);
                tri_normal64(v, n);
                // hit point on the triangle's plane
                const double dn = d[0] * n[0] + d[1] * n[1] + d[2] * n[2];
                const double th = ((v[0] - o[0]) * n[0] + (v[1] - o[1]) * n[1] + (v[2] - o[2]) * n[2]) / dn;
                double x[3];
                for (int c = 0; c < 3; c++) x[c] = o[c] + th * d[c];
                const int side = dn < 0.0 ? 0 : 1;
                const double sg = side ? -1.0 : 1.0;
                const unsigned mt = B.tri_mat[B.part[p].tri_begin + tl];
                const int mi = side ? (int)(mt >> 16) : (int)(mt & 0xffffu);
                const double rs = B.mat64[2 * mi], rd = B.mat64[2 * mi + 1];
                if (rd > 0.0) {
                    DEmit &e = out[ne++];
                    for (int c = 0; c < 3; c++) { e.x[c] = x[c]; e.nf[c] = sg * n[c]; }
                    e.wd = wgt * rd / K;
                    e.src = h;
                    e.c0 = ((unsigned long long)ray * (unsigned long long)nseg + (unsigned long long)k) *
                           (unsigned long long)K;
                }
                wgt *= rs;
                if (wgt == 0.0) break;
                for (int c = 0; c < 3; c++) { d[c] = d[c] - 2.0 * dn * n[c]; o[c] = x[c]; }
            }
        }
        cnt[ray] = ne;
    }
}

// Step 2: a block per slot turns the per-ray record counts into
// their exclusive prefix (each thread a contiguous range, then the block's
// ranges in order) and the slot's total.
__global__ void __launch_bounds__(1024) k_dscan(TraceArgs a)
{
    pdl_enter();
    __shared__ int part[1024];
    const int s = blockIdx.x;
    const size_t R = (size_t)a.sd[s].N * a.sd[s].N;
    int *cnt = a.dcnt + (size_t)s * a.ray_stride;
    const size_t per = (R + blockDim.x - 1) / blockDim.x;
    const size_t r0 = min(R, per * threadIdx.x), r1 = min(R, r0 + per);
    int sum = 0;
    for (size_t r = r0; r < r1; r++) sum += cnt[r];
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < (int)blockDim.x; o <<= 1) {  // inclusive scan of the ranges' sums
        const int v = threadIdx.x >= (unsigned)o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    int run = part[threadIdx.x] - sum;
    for (size_t r = r0; r < r1; r++) {
        const int c = cnt[r];
        cnt[r] = run;
        run += c;
    }
    if (threadIdx.x == blockDim.x - 1) a.dtot[s] = part[threadIdx.x];
}

// Step 3: a thread per (record, sample) work item, items in the
// order of the records (ray-major), each record's K samples consecutive; the
// record of item e K + q is found by binary search over the prefix.
// (four blocks an SM, 128 registers, 144 B of spills: 3.08 ms against 3.57 at three and 3.50 at five, at 64 blocks a
// slot)
__global__ void __launch_bounds__(kLaneStride, 4) k_diffuse(TraceArgs a)
{
    pdl_enter();
    __shared__ TraceCtx B;
    __shared__ double red[4][6];
    __shared__ __align__(16) WalkShared s_walk[kLaneStride / 32];
    const int s = blockIdx.y;
    if ((size_t)blockIdx.x * blockDim.x >= (size_t)a.dtot[s] * (size_t)a.n_diffuse) {  // no items (uniform)
        if (threadIdx.x < 6) a.dpart[((size_t)s * kDiffBlocks + blockIdx.x) * 6 + threadIdx.x] = 0.0;
        return;
    }
    load_ctx(B, a, s);
    __syncthreads();
    double acc[6] = {0, 0, 0, 0, 0, 0};
    if (!B.skip) {
        const SlotDesc &D = a.sd[s];
        const int N = D.N, nseg = D.nseg, K = a.n_diffuse;
        const size_t R = (size_t)N * N;
        const int *off = a.dcnt + (size_t)s * a.ray_stride;
        const DEmit *rec = a.demit + (size_t)s * a.ray_stride * (size_t)(nseg - 1);
        int flags = 0;
        const size_t items = (size_t)a.dtot[s] * (size_t)K;
        // (every lane of a warp runs the same iterations: the walk is the warp's)
        for (size_t it0 = (size_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); it0 < items;
             it0 += (size_t)gridDim.x * blockDim.x) {
            const size_t it = it0 + (threadIdx.x & 31u);
            const bool live = it < items;
            const int e = live ? (int)(it / K) : 0;
            const int q = (int)(it - (size_t)e * K);
            const DEmit *E = rec;
            if (live) {
                // the last ray whose first record is <= e
                size_t lo = 0, hi = R - 1;
                while (lo < hi) {
                    const size_t mid = (lo + hi + 1) >> 1;
                    if (__ldg(off + mid) <= e) lo = mid; else hi = mid - 1;
                }
                E = rec + lo * (size_t)(nseg - 1) + (size_t)(e - __ldg(off + lo));
            }
            __syncwarp();
            diffuse_sample(B, s_walk[threadIdx.x >> 5], D.mesh, live, (unsigned long long)a.diffuse_seed,
                           live ? E->c0 + (unsigned long long)q : 0ull, E->x, E->nf, live ? E->src : -1,
                           live ? E->wd : 0.0, acc, flags);
            __syncwarp();
        }
        if (flags) atomicOr(&a.pose[s].flags, flags);
    }
    // block sum in a fixed order: warps by shuffles, then the four warps in turn
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double sum = warp_sums<6>(acc, lane);
    const int kv = warp_sum_value<6>(lane);
    if (kv >= 0) red[w][kv] = sum;
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        a.dpart[((size_t)s * kDiffBlocks + blockIdx.x) * 6 + k] = ((red[0][k] + red[1][k]) + red[2][k]) + red[3][k];
    }
}

// ------------------------------------------------------------- reduce
// First level: block b of slot s sums tiles [b * chunk, (b + 1) * chunk), and
// re-traces in FP64 the rays its tiles handed off (a walk bound, or more
// uncertain triangles than the candidate list holds; rare: the traversal
// context is loaded only when the block has any).  Each thread takes a fixed,
// strided set of tiles in order, so the sums are reproducible.
__device__ void final_reduce(const TraceArgs &a, int s, int eval0, double *force, double *torque, int *err_flags,
                             unsigned long long *stats_accum, bool cg);

// Re-traced rays of a block that its warps take one by one (nearest64_warp); with more, a lane
// a ray.  A warp takes 40-60 us a ray and a block has eight warps; a lane takes 100-350 us, but
// up to 32 of them run at once: the two meet near four rays a warp.
constexpr int kWarpRays = 32;
// Warps of a first-level block, resident blocks: 32 box-wing evaluations a launch 39 us at two
// blocks an SM (128 registers), 32.6 at four (the re-trace, rarely run, spills 372 B), 31.6 at five.
constexpr int kRedWarps = 8, kRedBlocksPerSM = 4;

struct RefineShared {
    int n[kRedWarps], first[32 * kRedWarps];
    double sum[kRedWarps][kPart];
    Walk64 walk[kRedWarps];
};

// The re-trace of the rays that tiles [t0, t1) of slot s handed off, summed by the
// thread that owns the tile into its acc.  (Out of line: rare, and its registers are not
// the reduction's.)  200k triangles, 1024^2, two bounces, eight evaluations: 366 -> 131 us
// where rays overflow, a warp a ray against a lane a ray.
__device__ __noinline__ void refine_block(const TraceCtx &B, const TraceArgs &a, int s, int t0, int t1, size_t base,
                                          RefineShared &S, double *acc, int &flags)
{
    // the block's rays in the order of its threads: own of them from first
    int own = 0;
    for (int t = t0 + (int)threadIdx.x; t < t1; t += blockDim.x) own += a.amb_count[base + t];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int first = own;
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, first, o);
        if (lane >= o) first += x;
    }
    if (lane == 31) S.n[w] = first;
    __syncthreads();
    int total = 0;
    for (int q = 0; q < kRedWarps; q++) {
        if (q == w) first += total - own;
        total += S.n[q];
    }
    if (total <= kWarpRays) {
        // few: a warp a ray, added by the owners in their order
        S.first[threadIdx.x] = first;
        for (int r0 = 0; r0 < total; r0 += kRedWarps) {
            __syncthreads();
            const int ray = r0 + w;
            if (ray < total) {
                int o = 0;  // the last thread that starts at or before it
                for (int h = kRedWarps * 16; h; h >>= 1)
                    if (S.first[o + h] <= ray) o += h;
                int q = ray - S.first[o], t = t0 + o;
                for (int c; q >= (c = a.amb_count[base + t]); t += blockDim.x) q -= c;
                double x[kPart];
                for (int k = 0; k < kPart; k++) x[k] = 0.0;
                refine_ray(B, a, s, a.amb_list[(base + t) * kTileRays + q], &S.walk[w], x, flags);
                if (lane == 0)
                    for (int k = 0; k < kPart; k++) S.sum[w][k] = x[k];
            }
            __syncthreads();
            for (int q = 0; q < kRedWarps; q++)
                if (r0 + q >= first && r0 + q < first + own)
                    for (int k = 0; k < kPart; k++) acc[k] += S.sum[q][k];
        }
    } else {
        for (int t = t0 + (int)threadIdx.x; t < t1; t += blockDim.x) {
            const int n = a.amb_count[base + t];
            for (int q = 0; q < n; q++) refine_ray(B, a, s, a.amb_list[(base + t) * kTileRays + q], nullptr, acc, flags);
        }
    }
}

// The outputs of an evaluation that was not run: zero force and torque, or NaN (and its rays
// counted, each a segment without a hit) where it had no Sun direction.
__device__ __forceinline__ void skipped_outputs(const TraceArgs &a, int s, int eval0, double *force, double *torque,
                                                unsigned long long *stats_accum)
{
    const bool dir = a.pose[s].skip == kSkipDir;
    if (threadIdx.x < 6) (threadIdx.x < 3 ? force : torque)[3 * (eval0 + s) + threadIdx.x % 3] = dir ? (double)NAN : 0.0;
    if (dir && stats_accum && threadIdx.x == 0) {
        const unsigned long long N = (unsigned long long)a.sd[s].N;
        atomicAdd(&stats_accum[0], 1ull);
        atomicAdd(&stats_accum[1], N * N);
        atomicAdd(&stats_accum[3], N * N);
    }
}

__global__ void __launch_bounds__(32 * kRedWarps, kRedBlocksPerSM) k_reduce1(TraceArgs a, int eval0, double *force, double *torque,
                                                 int *err_flags, unsigned long long *stats_accum, int fuse)
{
    pdl_enter();
    const int s = blockIdx.y, b = blockIdx.x;
    if (a.pose[s].skip) {  // uniform over the block
        if (fuse && b == 0) skipped_outputs(a, s, eval0, force, torque, stats_accum);
        return;
    }
    const int nt = a.sd[s].tiles;
    const int chunk = (nt + kRed1 - 1) / kRed1;
    const int t0 = b * chunk, t1 = min(t0 + chunk, nt);
    const size_t base = (size_t)s * a.n_blocks_x;
    double f[6] = {0, 0, 0, 0, 0, 0};
    Comp32 f32[6];  // the FP32 sum modes
    for (int k = 0; k < 6; k++) f32[k] = Comp32{0.0f, 0.0f};
    const int mode = a.sum_mode;
    // hand-offs, segments and hits of one block (at most 32768 tiles of 32 rays) fit 32 bits
    unsigned c[kCntRay];
    for (int k = 0; k < kCntRay; k++) c[k] = 0u;
    int mine = 0;
    for (int t = t0 + (int)threadIdx.x; t < t1; t += blockDim.x) {
        const float2 *pp = reinterpret_cast<const float2 *>(a.partials + (base + t) * 6);
        const float2 p2[3] = {pp[0], pp[1], pp[2]};
        for (int k = 0; k < 6; k++) {
            const float p = k & 1 ? p2[k >> 1].y : p2[k >> 1].x;
            if (mode == 0) f[k] += (double)p;
            else if (mode == 1) comp_add(f32[k], p);
            else f32[k].hi = __fadd_rn(f32[k].hi, p);
        }
        // count 0: the tile's hand-off flags; the re-trace below counts the rays it does
        for (int k = 1; k < kCntRay; k++) c[k] += a.pcounts[(base + t) * kCnt + k];
        mine |= a.amb_count[base + t];
    }
    __shared__ TraceCtx B;
    __shared__ int blk_flags;
    __shared__ union {  // (40 KB side by side made a launch of eight evaluations 2 us slower)
        RefineShared re;
        Comp32 r32[6][32 * kRedWarps];
    } sh;
    if (__syncthreads_or(mine)) {
        if (threadIdx.x == 0) blk_flags = 0;
        load_ctx(B, a, s);
        __syncthreads();
        int flags = 0;
        double acc[kPart];
        for (int k = 0; k < kPart; k++) acc[k] = 0.0;
        refine_block(B, a, s, t0, t1, base, sh.re, acc, flags);
        for (int k = 0; k < 6; k++) {
            if (mode == 0) f[k] += acc[k];
            else if (mode == 1) comp_add(f32[k], (float)acc[k]);
            else f32[k].hi = __fadd_rn(f32[k].hi, (float)acc[k]);
        }
        for (int k = 0; k < kCntRay; k++) c[k] += (unsigned)acc[6 + k];
        if (flags) atomicOr(&blk_flags, flags);
        __syncthreads();
        if (threadIdx.x == 0 && blk_flags) atomicOr(&a.pose[s].flags, blk_flags);
    }
    // block sums in a fixed order: FP64 for force and torque (or the FP32
    // modes' sums, threads in turn by one thread), integers for counts
    __shared__ double rf[6][8];
    __shared__ unsigned long long rc[kCnt][8];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (mode == 0) {
        const double x = warp_sums<6>(f, lane);
        const int k = warp_sum_value<6>(lane);
        if (k >= 0) rf[k][w] = x;
    } else {
        for (int k = 0; k < 6; k++) sh.r32[k][threadIdx.x] = f32[k];
    }
    for (int k = 0; k < kCntRay; k++) {
        const unsigned x = __reduce_add_sync(0xffffffffu, c[k]);
        if (lane == 0) rc[k][w] = x;
    }
    // the traversal counters, which the trace writes only when counting: thousands of nodes a ray pass 32 bits
    for (int k = kCntRay; k < kCnt; k++) {
        unsigned long long x = 0ull;
        if (a.count) {
            for (int t = t0 + (int)threadIdx.x; t < t1; t += blockDim.x) x += a.pcounts[(base + t) * kCnt + k];
            for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        }
        if (lane == 0) rc[k][w] = x;
    }
    __syncthreads();
    const int nw = (int)(blockDim.x >> 5);
    double *out = a.partials1 + ((size_t)s * kRed1 + b) * kPart;
    if (threadIdx.x < 6) {
        if (mode == 0) {
            double x = 0.0;
            for (int q = 0; q < nw; q++) x += rf[threadIdx.x][q];
            out[threadIdx.x] = x;
        } else {
            Comp32 x{0.0f, 0.0f};
            for (int q = 0; q < (int)blockDim.x; q++) {
                if (mode == 1) comp_merge(x, sh.r32[threadIdx.x][q]);
                else x.hi = __fadd_rn(x.hi, sh.r32[threadIdx.x][q].hi);
            }
            out[threadIdx.x] = (double)comp_value(x);  // an FP32 value, exact in FP64
        }
    } else if (threadIdx.x < kPart) {
        unsigned long long x = 0ull;
        for (int q = 0; q < nw; q++) x += rc[threadIdx.x - 6][q];
        out[threadIdx.x] = __longlong_as_double((long long)x);  // (an integer's bits)
    }
    if (!fuse) return;
    // the last of the slot's blocks to finish adds the first-level sums, in
    // block order whichever block that is (the second level, without a launch)
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&a.red_ticket[s], 1u) == (unsigned)(kRed1 - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    final_reduce(a, s, eval0, force, torque, err_flags, stats_accum, true);
}

// The second level for slot s: its kRed1 first-level sums added by warps in a
// fixed tree (FP64; the FP32 modes add them again in FP32, in block order), the
// diffuse blocks' sums in block order, the pixel-area scale, the stores.  The
// calling block has kRed1 threads at least; `cg` reads what other blocks of the
// same launch wrote through L2.  The first warps sum the forces, the last one forms
// the scale beside them, and the counts (whole numbers) are added by every warp:
// the FP64 chain after the last block's arrival is 8 + kRed1 / 32 additions and a
// product (100 additions a warp and a serial tail, 18 us a launch of one slot, before).
// stats_accum[16]: 0 evals, 1 rays, 2 refined rays, 3 segments, 4..8 hits per segment,
// 9 nodes, 10 triangles, 11 box tests, 12..15 hand-offs by cause.
__device__ void final_reduce(const TraceArgs &a, int s, int eval0, double *force, double *torque, int *err_flags,
                             unsigned long long *stats_accum, bool cg)
{
    __shared__ double red2[6][kRed1 / 32];
    __shared__ double s_scale;
    __shared__ double diff[6][kDiffSums];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (int)(blockDim.x >> 5);
    const auto first = [&](int b, int k) {
        const double *src = a.partials1 + ((size_t)s * kRed1 + b) * kPart + k;
        return cg ? __ldcg(src) : *src;
    };
    if (a.n_diffuse > 0 && threadIdx.x < kDiffSums)
        for (int k = 0; k < 6; k++) {
            double x = 0.0;
            for (int b = threadIdx.x; b < kDiffBlocks; b += kDiffSums) x += a.dpart[((size_t)s * kDiffBlocks + b) * 6 + k];
            diff[k][threadIdx.x] = x;
        }
    if (w < kRed1 / 32) {
        double v[6];
        for (int k = 0; k < 6; k++) v[k] = first(threadIdx.x, k);
        const double x = warp_sums<6>(v, lane);
        const int k = warp_sum_value<6>(lane);
        if (k >= 0) red2[k][w] = x;
    }
    if (w == nw - 1) {
        const SlotPose &P = a.pose[s];
        const int N = a.sd[s].N;
        const double Du = ord_to_dbl(P.wmax_bits[0]) - ord_to_dbl(P.wmin_bits[0]);
        const double Dv = ord_to_dbl(P.wmax_bits[1]) - ord_to_dbl(P.wmin_bits[1]);
        const double sc = P.scale * (Du * Dv) / ((double)N * (double)N);
        if (lane == 0) {
            s_scale = sc;
            const int pflags = cg ? __ldcg(&P.flags) : P.flags;
            if (pflags) atomicOr(err_flags, pflags);
            if (stats_accum) {
                atomicAdd(&stats_accum[0], 1ull);
                atomicAdd(&stats_accum[1], (unsigned long long)N * (unsigned long long)N);
            }
        }
    }
    if (stats_accum) {
        for (int k = nw - 1 - w; k < kCnt; k += nw) {
            unsigned long long x = 0ull;
            for (int b = lane; b < kRed1; b += 32) x += (unsigned long long)__double_as_longlong(first(b, 6 + k));
            for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0 && x) atomicAdd(&stats_accum[2 + k], x);
        }
    }
    __syncthreads();
    if (threadIdx.x >= 6) return;
    const int k = threadIdx.x;
    double x = 0.0;
    if (a.sum_mode == 0) {
        for (int q = 0; q < kRed1 / 32; q++) x += red2[k][q];
        if (a.n_diffuse > 0)
            for (int g = 0; g < kDiffSums; g++) x += diff[k][g];
    } else {
        // the FP32 modes: the first-level sums again, in order, in FP32
        Comp32 y{0.0f, 0.0f};
        const auto add = [&](float p) {
            if (a.sum_mode == 1) comp_add(y, p);
            else y.hi = __fadd_rn(y.hi, p);
        };
        for (int b = 0; b < kRed1; b++) add((float)first(b, k));
        if (a.n_diffuse > 0)
            for (int g = 0; g < kDiffSums; g++) add((float)diff[k][g]);
        x = (double)comp_value(y);
    }
    (k < 3 ? force : torque)[3 * (eval0 + s) + k % 3] = x * s_scale;
}

// The second level as its own launch (after the diffuse rays), a block per slot.
__global__ void __launch_bounds__(kRed1) k_reduce(TraceArgs a, int eval0, double *force, double *torque, int *err_flags,
                                                unsigned long long *stats_accum)
{
    pdl_enter();
    const int s = blockIdx.x;
    if (a.pose[s].skip) {
        skipped_outputs(a, s, eval0, force, torque, stats_accum);
        return;
    }
    final_reduce(a, s, eval0, force, torque, err_flags, stats_accum, false);
}

// ------------------------------------------------------------ BVH check
// One thread per part walks the part's 4-wide tree of slot 0 from the root:
// every child box of a reached node must lie inside the box its parent holds
// for that node (the root's inside the part's root box), every leaf
// triangle's three vertices inside its leaf box; each leaf reference is
// counted per triangle.  report: [0] leaf references, [2] child boxes outside
// the parent's, [3] leaf triangles outside their box, [4] nodes reached,
// [5] walks stopped by their bound ([1], [6], [7] are filled on the host).
__global__ void k_bvh_check(const unsigned char *tctx, int *tri_seen, unsigned long long *report)
{
    const TraceCtx &B = *reinterpret_cast<const TraceCtx *>(tctx);
    const PartView &pv = B.part[blockIdx.x];
    if (threadIdx.x != 0 || !(pv.box_src[0] < INFINITY)) return;  // (a part without triangles)
    unsigned long long refs = 0, outside_box = 0, outside_tri = 0, nodes = 0, bound = 0;
    auto inside = [](const float *in, const float *out) {
        return in[0] >= out[0] && in[1] <= out[1] && in[2] >= out[2] && in[3] <= out[3] && in[4] >= out[4] &&
               in[5] <= out[5];
    };
    auto tri_inside = [&](int tl, const float *bx) {
        const float4 *tr = pv.tri + (size_t)tl * 3;
        bool ok = true;
        for (int c = 0; c < 3; c++) {
            const float4 v = tr[c];
            ok = ok && v.x >= bx[0] && v.x <= bx[1] && v.y >= bx[2] && v.y <= bx[3] && v.z >= bx[4] && v.z <= bx[5];
        }
        atomicAdd(tri_seen + pv.tri_begin + tl, 1);
        refs++;
        if (!ok) outside_tri++;
    };
    const float *bs = pv.box_src;
    const float root_box[6] = {bs[0], bs[3], bs[1], bs[4], bs[2], bs[5]};
    if (pv.root < 0) {
        tri_inside(~pv.root, root_box);
    } else {
        // stack of (node, parent slot box) pairs: the box is re-read from the parent node
        constexpr int kCheckStack = 256;
        int st_node[kCheckStack], st_par[kCheckStack];
        int sp = 0, iters = 0;
        st_node[sp] = pv.root;
        st_par[sp] = -1;
        sp++;
        const int limit = pv.limit;
        while (sp > 0) {
            if (++iters > limit) { bound++; break; }
            sp--;
            const int nd = st_node[sp], par = st_par[sp];
            float pbox[6];
            if (par < 0) {
                for (int k = 0; k < 6; k++) pbox[k] = root_box[k];
            } else {
                const float4 *pn = pv.node + (size_t)(par >> 2) * kNode4;
                const int c = par & 3;
                for (int k = 0; k < 6; k++) pbox[k] = reinterpret_cast<const float *>(pn + k)[c];
            }
            const float4 *n = pv.node + (size_t)nd * kNode4;
            const int4 refs4 = *reinterpret_cast<const int4 *>(n + 6);
            const int rf[4] = {refs4.x, refs4.y, refs4.z, refs4.w};
            nodes++;
            const int used = reinterpret_cast<const int4 *>(n + 7)->z;  // (the children come first)
            for (int c = 0; c < used; c++) {
                float bx[6];
                for (int k = 0; k < 6; k++) bx[k] = reinterpret_cast<const float *>(n + k)[c];
                if (!inside(bx, pbox)) outside_box++;
                if (rf[c] >= 0) {
                    if (sp >= kCheckStack) { bound++; continue; }
                    st_node[sp] = rf[c];
                    st_par[sp] = nd * 4 + c;
                    sp++;
                } else {
                    tri_inside(~rf[c], bx);
                }
            }
        }
    }
    atomicAdd(report + 0, refs);
    atomicAdd(report + 2, outside_box);
    atomicAdd(report + 3, outside_tri);
    atomicAdd(report + 4, nodes);
    atomicAdd(report + 5, bound);
}

cudaError_t launch_bvh_check(const unsigned char *tctx, int n_parts, int *tri_seen, unsigned long long *report,
                             cudaStream_t st)
{
    k_bvh_check<<<n_parts, 32, 0, st>>>(tctx, tri_seen, report);
    return cudaGetLastError();
}

// ------------------------------------------------------------ launchers
// All-ones pixel keys (no hit, no candidate) before the first raster pass.
__global__ void __launch_bounds__(256) k_clear_keys(unsigned long long *key, size_t n)
{
    pdl_enter();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        key[i] = ~0ull;
}

static int device_sms()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    return std::max(1, sms);
}

int raster_launches(int S, bool queue)
{
    if (few_slots(S)) return queue ? 3 : 4;  // first pass, chunk listing, chunks; the merged second pass
    return queue ? 4 : 6;                     // key clear, first pass, listing, chunks; two second-pass launches
}

cudaError_t launch_frame(const TraceArgs &a, int S, cudaStream_t st)
{
    const int sms = device_sms();
    const bool raster = a.raster && a.rast_tris > 0 && a.n_tiles > 0;
    const bool few = few_slots(S);
    TraceArgs f = a;
    if (!raster || !few) f.pix_key = nullptr;
    cudaError_t e;
    if (raster && few) {
        // the frame kernel's blocks beyond the context's warp clear the pixel keys
        const size_t per = (size_t)256 * 4;  // keys a block clears in one sweep of four
        const int ky = (int)std::max<size_t>(1, std::min((a.ray_stride + per - 1) / per,
                                                         (size_t)(sms * 4 + S - 1) / (size_t)S));
        e = launch_chained(k_frame, dim3(S, ky), dim3(256), 0, st, f);
    } else {
        e = launch_chained(k_frame, dim3(S, 1), dim3(32), 0, st, f);
    }
    if (e != cudaSuccess || !raster) return e;
    if (!few) {
        const size_t px = (size_t)S * a.ray_stride;
        const size_t kb = std::min((px + 255) / 256, (size_t)sms * 8);
        e = launch_chained(k_clear_keys, dim3((unsigned)std::max<size_t>(1, kb)), dim3(256), 0, st, a.pix_key, px);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((a.rast_tris + 127) / 128, S);
    // the chunk lists grow with the slots: a grid of the device's size per eight
    // slots, not of the lists' capacity
    const int big_blocks = sms * kRastBigBlocksPerSM * std::max(1, (S + 7) / 8);
    if ((e = launch_chained(k_raster<0>, grid, dim3(128), 0, st, a)) != cudaSuccess) return e;
    if ((e = launch_chained(k_raster_chunks, dim3(std::max(1, big_blocks / 4)), dim3(256), 0, st, a)) != cudaSuccess)
        return e;
    if ((e = launch_chained(k_raster_big<0>, dim3(big_blocks), dim3(256), 0, st, a)) != cudaSuccess) return e;
    if (a.queue) return cudaSuccess;  // the work queue runs the second pass with the trace
    if (few) {
        // the second pass over large triangles' chunks and small triangles: one launch
        const int nbig = 2 * big_blocks, per_slot = (int)grid.x;
        const unsigned blocks = (unsigned)nbig + (unsigned)per_slot * (unsigned)S;
        return launch_chained(k_raster_pass1, dim3(blocks), dim3(128), 0, st, a, nbig, per_slot);
    }
    if ((e = launch_chained(k_raster<1>, grid, dim3(128), 0, st, a)) != cudaSuccess) return e;
    return launch_chained(k_raster_big<1>, dim3(big_blocks), dim3(256), 0, st, a);
}

// The trace kernels' split of the SM's 256 KB between L1 and shared memory:
// a request for a small shared-memory configuration, so that L1 keeps most of
// the SM's memory for the hot tree nodes and the traversal stacks.  The
// driver's default had been 132 KB of shared memory (L1 124 KB); with this
// request and the context and hit columns sized per launch (7.4 KB a block of
// the headline workload) it takes 100 KB for the eight blocks the registers
// allow (L1 156 KB, L1 hit rate 68 -> 74%).  A percentage of the largest
// shared-memory configuration (228 KB); the driver rounds it up to a
// configuration that holds the blocks.
constexpr int kTraceCarveoutPct = 27;

cudaError_t configure_trace_kernels()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, kTraceCarveoutPct);
    };
    set((const void *)k_trace<false, false>);
    set((const void *)k_trace<false, true>);
    set((const void *)k_trace<true, false>);
    set((const void *)k_trace<true, true>);
    set((const void *)k_queue<false, false>);
    set((const void *)k_queue<false, true>);
    set((const void *)k_queue<true, false>);
    set((const void *)k_queue<true, true>);
    return e;
}

cudaError_t launch_trace(const TraceArgs &a, int S, cudaStream_t st)
{
    (void)S;
    if (a.n_tiles <= 0) return cudaSuccess;
    // the hit records and the traversal counters are separate kernel variants:
    // code a launch never runs still costs registers in the others
    const dim3 g(a.n_tiles), b(kTileRays * kTraceWarps);
    const size_t dyn = trace_dyn_bytes(a.ctx_parts, a.hpt_segs);
    if (a.queue) {
        // persistent: as many blocks as fit on the device at once
        const dim3 gq(device_sms() * kQueueBlocksPerSM);
        if (a.count) return launch_chained(a.hits ? k_queue<true, true> : k_queue<true, false>, gq, b, dyn, st, a);
        return launch_chained(a.hits ? k_queue<false, true> : k_queue<false, false>, gq, b, dyn, st, a);
    }
    if (a.few_tiles > 0 && !a.count)
        return launch_chained(a.hits ? k_trace_few<true> : k_trace_few<false>, dim3(a.few_tiles), dim3(32 * kFewWarps), 0, st, a);
    if (a.count) return launch_chained(a.hits ? k_trace<true, true> : k_trace<true, false>, g, b, dyn, st, a);
    return launch_chained(a.hits ? k_trace<false, true> : k_trace<false, false>, g, b, dyn, st, a);
}

cudaError_t launch_reduce(const TraceArgs &a, int S, int eval0, double *force, double *torque, int *err_flags,
                          unsigned long long *stats_accum, cudaStream_t st)
{
    // without diffuse rays the last first-level block of a slot does the second level
    const int fuse = (a.n_diffuse <= 0 && a.red_ticket) ? 1 : 0;
    cudaError_t e = launch_chained(k_reduce1, dim3(kRed1, S), dim3(32 * kRedWarps), 0, st, a, eval0, force, torque, err_flags,
                                   stats_accum, fuse);
    if (e != cudaSuccess || fuse) return e;
    // diffuse secondaries after the FP64 re-trace (which records the hits of the rays it takes)
    if (a.n_diffuse > 0) {
        if ((e = launch_chained(k_demit, dim3(kDiffBlocks, S), dim3(kLaneStride), 0, st, a)) != cudaSuccess) return e;
        if ((e = launch_chained(k_dscan, dim3(S), dim3(1024), 0, st, a)) != cudaSuccess) return e;
        if ((e = launch_chained(k_diffuse, dim3(kDiffBlocks, S), dim3(kLaneStride), 0, st, a)) != cudaSuccess) return e;
    }
    return launch_chained(k_reduce, dim3(S), dim3(kRed1), 0, st, a, eval0, force, torque, err_flags, stats_accum);
}

}  // namespace srp
