// Device code of the photon tracker (sm_103a).
//
//  * k_trace, k_trace_few: closest hits of given rays (the geometry query alone).
//  * k_sample_source:  first photon state from a source (one photon per lane).
//  * k_propagate:      persistent kernel; the photons of a CTA wait in slots in
//                      shared memory for one of four kinds of work (query of
//                      the geometry, bulk event, surface event, tally and
//                      rebirth), and each warp takes a batch of one kind (see
//                      there).  Photon ids come from a global atomic work
//                      queue; fate tallies live in shared memory per CTA;
//                      per-channel counts and the time histogram use global
//                      atomics.  Template builds <kStats, kAdjoint, kSpectral>
//                      add traversal counters, the adjoint tallies, and a
//                      wavelength carried by each photon (dispersion); the
//                      default build <0,0,0> has none of them.
//
// Bit-exactness of the closest hit: the triangle test below performs the same
// IEEE float operations, in the same order, as a plain C implementation of
// the watertight test (Woop, Benthin & Wald, JCGT 2013); every operation is an
// explicit round-to-nearest intrinsic so the compiler cannot contract or
// reorder it.  Boxes are widened at build time and the box test uses a
// relative slack, so the traversal visits every box that holds a candidate;
// the walk through the grid passes every cell that holds a part of one.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "lxo_internal.h"

namespace lxo {

#define FULL_MASK 0xFFFFFFFFu
// Checked build (a substitute for a memory checker): every BVH node,
// triangle record, cell and tally row index is compared with its array size
// before use; a bad one sets kErrBounds and ends the ray or skips the write,
// never an out-of-range access.  Compiled out by default.
#ifndef LXO_CHECK_BOUNDS
#define LXO_CHECK_BOUNDS 0
#endif

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11)
// ---------------------------------------------------------------------------
struct U4 {
    float u0, u1, u2, u3;
};

// kRounds: rounds per iteration of the code.  10, no loop, is fastest by
// itself; the photon loop uses 2 (and 1 where it is not hot), since long code
// costs it more than the loop: 1e6 photons of the DARWIN-scale mesh 4.75 -> 4.70
// ms, 2e7 63.5 -> 62.6, 3e6 of the 50 cm TPC 11.4 -> 11.2.
template <int kRounds = 2>
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll kRounds
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

__device__ __forceinline__ float u01(uint32_t x)
{
    // ((x >> 9) + 0.5) * 2^-23: exact in float, in [2^-24, 1 - 2^-24]
    return __fmul_rn(__uint2float_rn(x >> 9) + 0.5f, 1.1920928955078125e-07f);
}

template <int kRounds = 2>
__device__ __forceinline__ U4 draw4(uint64_t seed, uint64_t pid, uint32_t step, uint32_t draw)
{
    uint4 o = philox4x32_10<kRounds>(make_uint4((uint32_t)pid, (uint32_t)(pid >> 32), step, draw),
                            make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    return U4{u01(o.x), u01(o.y), u01(o.z), u01(o.w)};
}

// ---------------------------------------------------------------------------
// small float3 helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float s, float3 a) { return f3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross(float3 a, float3 b)
{
    return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float3 normalize(float3 a) { return rsqrtf(dot(a, a)) * a; }

// orthonormal basis perpendicular to unit n (Duff et al., JCGT 6(1), 2017)
__device__ __forceinline__ void onb(float3 n, float3& t1, float3& t2)
{
    const float sgn = (n.z >= 0.0f) ? 1.0f : -1.0f;  // -0.0 counts as positive
    float a = -1.0f / (sgn + n.z);
    float b = n.x * n.y * a;
    t1 = f3(1.0f + sgn * n.x * n.x * a, sgn * b, -sgn * n.x);
    t2 = f3(b, sgn + n.y * n.y * a, -n.y);
}

// ---------------------------------------------------------------------------
// watertight ray / triangle test (exact op order, see file header)
// ---------------------------------------------------------------------------
struct WRay {
    float ox, oy, oz;
    float Sx, Sy, Sz;
    int kz;   // axis of the direction's largest component
};

__device__ __forceinline__ float pick(int k, float x, float y, float z) { return k == 0 ? x : (k == 1 ? y : z); }

// The axes kx, ky are not swapped for a negative component along kz: the swap
// negates U, V, W, det and T exactly, so every hit and t is the same.
__device__ __forceinline__ int shear(float3 d, float3& S)
{
    const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    const int kz = (ax >= ay) ? ((ax >= az) ? 0 : 2) : ((ay >= az) ? 1 : 2);
    const float dkz = pick(kz, d.x, d.y, d.z);
    S.x = __fdiv_rn(pick(kz, d.y, d.z, d.x), dkz);
    S.y = __fdiv_rn(pick(kz, d.z, d.x, d.y), dkz);
    S.z = __fdiv_rn(1.0f, dkz);
    return kz;
}

__device__ __forceinline__ WRay wray_setup(float3 o, float3 d)
{
    float3 S;
    const int kz = shear(d, S);
    return WRay{o.x, o.y, o.z, S.x, S.y, S.z, kz};
}

// The edge functions again in double, for when one of them rounded to zero
// in float (Woop et al.'s fallback).  Out of line: it is rarely taken, and
// inline it costs the hot leaf loop registers.
__device__ __noinline__ void edges_fp64(float Ax, float Ay, float Bx, float By, float Cx, float Cy, float& U, float& V,
                                        float& W)
{
    U = __double2float_rn(__dsub_rn(__dmul_rn((double)Cx, (double)By), __dmul_rn((double)Cy, (double)Bx)));
    V = __double2float_rn(__dsub_rn(__dmul_rn((double)Ax, (double)Cy), __dmul_rn((double)Ay, (double)Cx)));
    W = __double2float_rn(__dsub_rn(__dmul_rn((double)Bx, (double)Ay), __dmul_rn((double)By, (double)Ax)));
}

__device__ __forceinline__ bool wray_hit(const WRay& r, float4 a, float4 b, float4 c, float tmax, float& t_out)
{
    // vertices v0 = a.xyz, v1 = (a.w, b.x, b.y), v2 = (b.z, b.w, c.x)
    const float A0 = __fsub_rn(a.x, r.ox), A1 = __fsub_rn(a.y, r.oy), A2 = __fsub_rn(a.z, r.oz);
    const float B0 = __fsub_rn(a.w, r.ox), B1 = __fsub_rn(b.x, r.oy), B2 = __fsub_rn(b.y, r.oz);
    const float C0 = __fsub_rn(b.z, r.ox), C1 = __fsub_rn(b.w, r.oy), C2 = __fsub_rn(c.x, r.oz);
    // axes kx, ky = the two after kz in turn
    const bool k0 = r.kz == 0, k1 = r.kz == 1;
    const float Akz = k0 ? A0 : (k1 ? A1 : A2), Bkz = k0 ? B0 : (k1 ? B1 : B2), Ckz = k0 ? C0 : (k1 ? C1 : C2);
    const float Ax = __fsub_rn(k0 ? A1 : (k1 ? A2 : A0), __fmul_rn(r.Sx, Akz));
    const float Ay = __fsub_rn(k0 ? A2 : (k1 ? A0 : A1), __fmul_rn(r.Sy, Akz));
    const float Bx = __fsub_rn(k0 ? B1 : (k1 ? B2 : B0), __fmul_rn(r.Sx, Bkz));
    const float By = __fsub_rn(k0 ? B2 : (k1 ? B0 : B1), __fmul_rn(r.Sy, Bkz));
    const float Cx = __fsub_rn(k0 ? C1 : (k1 ? C2 : C0), __fmul_rn(r.Sx, Ckz));
    const float Cy = __fsub_rn(k0 ? C2 : (k1 ? C0 : C1), __fmul_rn(r.Sy, Ckz));
    float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    if (fminf(fminf(fabsf(U), fabsf(V)), fabsf(W)) == 0.0f) edges_fp64(Ax, Ay, Bx, By, Cx, Cy, U, V, W);
    if (fminf(fminf(U, V), W) < 0.0f && fmaxf(fmaxf(U, V), W) > 0.0f) return false;
    const float det = __fadd_rn(__fadd_rn(U, V), W);
    if (det == 0.0f) return false;
    const float Az = __fmul_rn(r.Sz, Akz), Bz = __fmul_rn(r.Sz, Bkz), Cz = __fmul_rn(r.Sz, Ckz);
    const float T = __fadd_rn(__fadd_rn(__fmul_rn(U, Az), __fmul_rn(V, Bz)), __fmul_rn(W, Cz));
    const float t = __fdiv_rn(T, det);
    if (!(t > 0.0f) || !(t <= tmax)) return false;
    t_out = t;
    return true;
}

// ---------------------------------------------------------------------------
// Closest hit with t in (0, tmax], skipping one triangle, ties to the smallest
// triangle id: layers entered by their cells, the rest of the scene walked
// through the grid (or searched by its main tree).
// ---------------------------------------------------------------------------
constexpr float kBoxSlack = 1.0f + 1.0f / 65536.0f;

// The reciprocal without IEEE rounding (1 ulp): the slab test is conservative
// by the boxes' margin and the slack, so the hits are the same.
__device__ __forceinline__ float fast_inv(float d)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fabsf(d) < 1e-20f ? 1e-20f : d));
    return r;
}

constexpr int kSlotF4 = 5;            // float4 per query slot in shared memory (see load_slot)
constexpr uint32_t kNoTri = 0x0FFFFFFFu;  // "no triangle" in 28 bits (ids stay below 2^28 - 1)

// Counting build: what one lane counts (warp-wide figures by lane 0).  Lane
// cycles by phase of the photon loop, a warp's clock times the lanes at work:
// node loop, leaf loop, traversal set-up (slots taken and read), random draws
// and the next flight, interaction, refill (tallies, new photons).
enum { kCycNode = 0, kCycLeaf, kCycBegin, kCycDraw, kCycFinish, kCycRefill, kCycPhases };

struct Counters {
    uint32_t steps, nodes, leaves, tris;
    uint32_t node_iters, leaf_iters, batches, entries, walks, walk_iters;
    uint32_t q_nodes, q_leaves;      // of the query in flight
    unsigned long long loop_cycles, idle_cycles;
    unsigned long long cyc[kCycPhases];
};

// The next triangle of a leaf, the leaf reference moved on past it (0 after the
// last); the closest triangle known by its record.  One triangle a call, since
// the lanes of a warp hold leaves of different sizes (all of a leaf at once
// ran 4.4 tests a call for 1.5 triangles a leaf).
__device__ __forceinline__ void triangle(const Scene& sc, const WRay& wr, uint32_t skip, int& leaf, float& bt,
                                         uint32_t& best_rec, int* bounds_err)
{
    const uint32_t enc = ~(uint32_t)leaf;
    const uint32_t r = enc >> 3;
    leaf = (enc & 7u) ? leaf - 7 : 0;   // (first + 1, count - 1): enc + 7
    if (LXO_CHECK_BOUNDS && r >= sc.n_records) {
        atomicOr(bounds_err, kErrBounds);
        return;
    }
    const float4* tr = sc.tris + 3 * (size_t)r;
    const float4 a = __ldg(tr + 0), b = __ldg(tr + 1), c = __ldg(tr + 2);
    const uint32_t id = __float_as_uint(c.y);
    float t;
    if (id != skip && wray_hit(wr, a, b, c, bt, t)) {
        // ties go to the smallest triangle id
        if (t < bt || best_rec == LXO_NO_HIT || id < __float_as_uint(__ldg(sc.tris + 3 * (size_t)best_rec + 2).y)) {
            bt = t;
            best_rec = r;
        }
    }
}

// Stack entries that are no leaf reference (those are above INT32_MIN + 6: < 2^28 records)
constexpr int kDone = INT32_MIN + 1;  // bottom of the stack
constexpr int kWalk = INT32_MIN + 2;  // back to the walk through the grid

__device__ __forceinline__ bool is_leaf(int node) { return (uint32_t)node > (uint32_t)kWalk; }

// Pushes the entries of the planar clusters in `mask` for a ray with t in
// (0, tmax]: a ray crossing the slab within a few grid cells starts at those
// cells' sub-trees; any other ray meeting the slab at the cluster root.
__device__ __forceinline__ void enter_clusters(const Scene& sc, uint32_t mask, float3 o, float3 d, float tmax,
                                               int* stack, int& sp)
{
    for (; mask; mask &= mask - 1) {
        const ClusterDev& cl = sc.clusters[__ffs(mask) - 1];
        const float oa = pick(cl.axis, o.x, o.y, o.z), ia = fast_inv(pick(cl.axis, d.x, d.y, d.z));
        const float ta = (cl.slab_lo - oa) * ia, tb = (cl.slab_hi - oa) * ia;
        const float tin = fmaxf(fminf(ta, tb), 0.0f), tout = fminf(fmaxf(ta, tb), tmax * kBoxSlack);
        if (!(tin <= tout)) continue;
        if (tout < 1e30f) {
            const int bu = cl.axis == 2 ? 0 : cl.axis + 1;   // in-plane axes (axis+1, axis+2) mod 3
            const int bv = cl.axis == 0 ? 2 : cl.axis - 1;
            const float ou = pick(bu, o.x, o.y, o.z), du = pick(bu, d.x, d.y, d.z);
            const float ov = pick(bv, o.x, o.y, o.z), dv = pick(bv, d.x, d.y, d.z);
            const float u1 = ou + tin * du, u2 = ou + tout * du, v1 = ov + tin * dv, v2 = ov + tout * dv;
            const float fi0 = fmaxf(floorf((fminf(u1, u2) - cl.delta - cl.u0) * cl.inv_cell), 0.0f);
            const float fi1 = fminf(floorf((fmaxf(u1, u2) + cl.delta - cl.u0) * cl.inv_cell), (float)(cl.nu - 1));
            const float fj0 = fmaxf(floorf((fminf(v1, v2) - cl.delta - cl.v0) * cl.inv_cell), 0.0f);
            const float fj1 = fminf(floorf((fmaxf(v1, v2) + cl.delta - cl.v0) * cl.inv_cell), (float)(cl.nv - 1));
            if (!(fi0 <= fi1) || !(fj0 <= fj1)) continue;  // outside the cluster's grid
            if ((fi1 - fi0 + 1.0f) * (fj1 - fj0 + 1.0f) <= (float)kMaxCellsPerRay) {
#pragma unroll 1
                for (int j = (int)fj0; j <= (int)fj1; ++j)
#pragma unroll 1
                    for (int i = (int)fi0; i <= (int)fi1; ++i) {
                        if (LXO_CHECK_BOUNDS && (i < 0 || j < 0 || i >= cl.nu || j >= cl.nv)) continue;
                        const int r = __ldg(&cl.cells[(size_t)j * cl.nu + i]);
                        if (r != kEmptyChild) stack[sp++] = r;
                    }
                continue;
            }
        }
        stack[sp++] = cl.root;
    }
}

// A ray for the slab test in grid space: i = 1 / direction, oi = origin * i.
struct RayInv {
    float ix, iy, iz, oix, oiy, oiz;
};

__device__ __forceinline__ RayInv ray_inv(const Scene& sc, float3 o, float3 d)
{
    RayInv r;
    r.ix = fast_inv(d.x) * sc.grid_h;
    r.iy = fast_inv(d.y) * sc.grid_h;
    r.iz = fast_inv(d.z) * sc.grid_h;
    r.oix = fmaf(o.x, sc.grid_inv, sc.grid_off[0]) * r.ix;
    r.oiy = fmaf(o.y, sc.grid_inv, sc.grid_off[1]) * r.iy;
    r.oiz = fmaf(o.z, sc.grid_inv, sc.grid_off[2]) * r.iz;
    return r;
}

// Where the slab tests of a caller's ray start.  From far away they are off by
// 5 to 7 x 2^-24 of the distance, which for small triangles passes the boxes'
// margin (2^-19 of the largest coordinate) from some 40 times that coordinate
// on: a ray that starts more than 192 cells from the grid's middle along some
// axis is moved along itself to 128 cells from there, still before the scene,
// which reaches 84.  The fma of the move rounds once, at the new place.  The
// tests then count their distance from there; their limits, which count from the
// origin, are larger than they need be, which is safe.  (The photon kernel tests
// from the photon's place: the same move in there, inline or out of line, took 3
// to 5 % of the time of all its runs.)
__device__ __forceinline__ float3 near_origin(const Scene& sc, float3 o, float3 d)
{
    const float3 g = f3(fmaf(o.x, sc.grid_inv, sc.grid_off[0]) - 49.0f, fmaf(o.y, sc.grid_inv, sc.grid_off[1]) - 49.0f,
                        fmaf(o.z, sc.grid_inv, sc.grid_off[2]) - 49.0f);
    const float m = fmaxf(fmaxf(fabsf(g.x), fabsf(g.y)), fabsf(g.z));
    if (!(m > 192.0f)) return o;
    // (scaled so that no square overflows; 1e-5: above the rounding here)
    const float dm = fmaxf(fmaxf(fabsf(d.x), fabsf(d.y)), fabsf(d.z));
    const float3 gs = __fdividef(1.0f, m) * g, ds = __fdividef(1.0f, dm) * d;
    const float cells = fmaf(m * (1.0f - 1e-5f), sqrtf(dot(gs, gs)), -128.0f);
    const float t = __fdividef(cells * sc.grid_h, dm * sqrtf(dot(ds, ds)));
    if (!(t < 1e30f)) return o;   // no direction, or numbers that do not carry it
    return f3(fmaf(t, d.x, o.x), fmaf(t, d.y, o.y), fmaf(t, d.z, o.z));
}

// State of a query: next node (kDone: finished), stack entries, axis kz,
// sub-tree of the last occupied cell, closest hit so far (t and record), and
// how far its walk has come.
struct Query {
    int node, sp, kz, seen;
    float bt, tw;
    uint32_t rec;
};

// Starts a query with t in (0, tmax]: the layers in `clusters` wait on the
// stack while the grid is walked from `clear` on (the main tree searched, if
// that is negative: the ray starts outside the grid).
__device__ __forceinline__ Query begin_query(const Scene& sc, float3 o, float3 d, int kz, float tmax, uint32_t clusters,
                                             float clear, int* stack)
{
    Query c{kWalk, 1, kz, kDone, tmax, clear, LXO_NO_HIT};
    stack[0] = kDone;
    if (clusters) enter_clusters(sc, clusters, o, d, tmax, stack, c.sp);
    if (!(clear >= 0.0f)) {
        c.node = sc.main_root;
        if (c.node == kEmptyChild) c.node = stack[--c.sp];
    }
    return c;
}

// One visit: the two children's boxes against the ray; descends into the
// nearer child hit and pushes the other, or pops.
__device__ __forceinline__ void node_visit(const Scene& sc, const RayInv& r, float lim, int& node, int* stack, int& sp,
                                           int* err)
{
    if (LXO_CHECK_BOUNDS && (uint32_t)node >= sc.n_nodes) {
        atomicOr(err, kErrBounds);
        node = kDone;
        sp = 1;
        return;
    }
    const float4* nd = sc.nodes + 4 * (size_t)node;
    const float4 nx = __ldg(nd + 0), ny = __ldg(nd + 1), nz = __ldg(nd + 2);
    const int4 cr = __ldg(reinterpret_cast<const int4*>(nd + 3));
    const float ax0 = fmaf(nx.x, r.ix, -r.oix), ax1 = fmaf(nx.y, r.ix, -r.oix);
    const float ay0 = fmaf(ny.x, r.iy, -r.oiy), ay1 = fmaf(ny.y, r.iy, -r.oiy);
    const float az0 = fmaf(nz.x, r.iz, -r.oiz), az1 = fmaf(nz.y, r.iz, -r.oiz);
    const float bx0 = fmaf(nx.z, r.ix, -r.oix), bx1 = fmaf(nx.w, r.ix, -r.oix);
    const float by0 = fmaf(ny.z, r.iy, -r.oiy), by1 = fmaf(ny.w, r.iy, -r.oiy);
    const float bz0 = fmaf(nz.z, r.iz, -r.oiz), bz1 = fmaf(nz.w, r.iz, -r.oiz);
    const float an = fmaxf(fmaxf(fminf(ax0, ax1), fminf(ay0, ay1)), fmaxf(fminf(az0, az1), 0.0f));
    const float af = fminf(fminf(fmaxf(ax0, ax1), fmaxf(ay0, ay1)), fminf(fmaxf(az0, az1), lim));
    const float bn = fmaxf(fmaxf(fminf(bx0, bx1), fminf(by0, by1)), fmaxf(fminf(bz0, bz1), 0.0f));
    const float bf = fminf(fminf(fmaxf(bx0, bx1), fmaxf(by0, by1)), fminf(fmaxf(bz0, bz1), lim));
    const bool ha = an <= af;
    const bool hb = bn <= bf;   // every node has two children (see the builder)
    const bool b_first = hb && !(ha && an <= bn);
    const int near = b_first ? cr.y : cr.x;
    if (ha && hb) {
        // lxo_build_bvh rejects a forest whose depth plus the <= 33 entries
        // the forest entry pushes could reach kStackSize, so this cannot
        // fire; only the checked build keeps the test (in the normal build
        // the never-taken exit cost 5 % of the time)
        if (LXO_CHECK_BOUNDS && sp >= kStackSize) {
            atomicOr(err, kErrStack);
            node = kDone;
            sp = 1;
            return;
        }
        stack[sp++] = b_first ? cr.x : cr.y;
    }
    node = near;
    if (!(ha || hb)) node = stack[--sp];
}

// Distance at which a ray leaves the cube of k cells (an octant's) that starts
// with its cell (x, y, z): in grid space, i = 1 / direction (large and positive
// for a ray along a side), oi = origin * i.
__device__ __forceinline__ float cube_exit(int x, int y, int z, float k, const RayInv& r)
{
    const float tx = fmaf(k, fabsf(r.ix), fmaf((float)x, r.ix, fminf(r.ix, 0.0f) - r.oix));
    const float ty = fmaf(k, fabsf(r.iy), fmaf((float)y, r.iy, fminf(r.iy, 0.0f) - r.oiy));
    const float tz = fmaf(k, fabsf(r.iz), fmaf((float)z, r.iz, fminf(r.iz, 0.0f) - r.oiz));
    return fminf(fminf(tx, ty), tz);
}

__device__ __forceinline__ uint32_t octant(const RayInv& r)
{
    return (__float_as_uint(r.ix) >> 31) | ((__float_as_uint(r.iy) >> 31) << 1) | ((__float_as_uint(r.iz) >> 31) << 2);
}

// How far a flight of length d from o along dir is clear by the walk grid's
// empty cubes: true if all of it is; else it is up to t, -1 if it starts
// outside the grid.  eps: a nudge past a cell's side, in t.
constexpr uint32_t kNoWalk = 0xFFFFu;   // that -1 where t is kept in 16 bits, in units of walk_unit

__device__ __forceinline__ bool clear_flight(const Scene& sc, float3 o, float3 dir, float d, const RayInv& r, float eps,
                                             float& t)
{
    t = -1.0f;
    if (!sc.walk_skip) return false;
    const float gx = fmaf(o.x, sc.grid_inv, sc.grid_off[0]), gy = fmaf(o.y, sc.grid_inv, sc.grid_off[1]),
                gz = fmaf(o.z, sc.grid_inv, sc.grid_off[2]);
    const float ux = dir.x * sc.grid_inv, uy = dir.y * sc.grid_inv, uz = dir.z * sc.grid_inv;
    const uint32_t oct = octant(r);
    float tc = 0.0f;
#pragma unroll 1
    for (int hop = 0; hop < kSafeHops; ++hop) {
        const int x = (int)fminf(fmaxf(fmaf(tc, ux, gx), 0.5f), sc.walk_max[0]);
        const int y = (int)fminf(fmaxf(fmaf(tc, uy, gy), 0.5f), sc.walk_max[1]);
        const int z = (int)fminf(fmaxf(fmaf(tc, uz, gz), 0.5f), sc.walk_max[2]);
        const uint32_t k = __ldg(&sc.walk_skip[8u * (uint32_t)((z * sc.walk_n[1] + y) * sc.walk_n[0] + x) + oct]);
        if (k == kCellOut) return hop > 0;   // it has left the grid: nothing is ahead
        t = tc;
        if (k == 0u) return false;
        tc = fmaxf(cube_exit(x, y, z, (float)k, r), tc) + eps;
        t = tc;
        if (tc > d) return true;
    }
    return false;
}

// One step of a query's walk through the grid: to the far side of the empty
// cube ahead, or of an occupied cell, whose sub-tree is descended first.  The
// triangles' parts reach over their cells by more than the nudge and the
// rounding here.  The walk is over (the next stack entry follows) once it has
// left the grid or passed the closest hit.
__device__ __forceinline__ void walk_step(const Scene& sc, const float4* q, const RayInv& r, float eps, float bt,
                                          float& t, int& node, int& seen, int* stack, int& sp, int* err)
{
    const float4 a = q[0], b = q[1];
    const int x = (int)fmaf(fmaf(t, b.x, a.x), sc.grid_inv, sc.grid_off[0]);
    const int y = (int)fmaf(fmaf(t, b.y, a.y), sc.grid_inv, sc.grid_off[1]);
    const int z = (int)fmaf(fmaf(t, b.z, a.z), sc.grid_inv, sc.grid_off[2]);
    // inside the grid by construction, which the checked build compares; the
    // limit guards the memory in the other
    if (LXO_CHECK_BOUNDS && ((uint32_t)x >= (uint32_t)sc.walk_n[0] || (uint32_t)y >= (uint32_t)sc.walk_n[1] ||
                             (uint32_t)z >= (uint32_t)sc.walk_n[2])) {
        atomicOr(err, kErrBounds);
        node = kDone;
        sp = 1;
        return;
    }
    const uint32_t c = min((uint32_t)((z * sc.walk_n[1] + y) * sc.walk_n[0] + x), sc.walk_cells - 1u);
    const uint32_t k = __ldg(&sc.walk_skip[8u * c + octant(r)]);
    if (k == 0u) {
        const int ref = __ldg(&sc.walk_ref[c]);
        if (ref != seen) {   // cells with the same triangles share a leaf
            node = seen = ref;
            stack[sp++] = kWalk;
        }
    }
    t = fmaxf(cube_exit(x, y, z, fmaxf((float)k, 1.0f), r), t) + eps;
    if (node == kWalk && (k == kCellOut || t > bt)) node = stack[--sp];
}

// Clusters whose slab the stretch of a ray with t in (0, tmax] may reach (bit
// c); the slabs are wider than the rounding here.
__device__ __forceinline__ uint32_t cluster_mask(const Scene& sc, float3 o, float3 d, float tmax)
{
    const float t = tmax * kBoxSlack;
    const float ex = fmaf(t, d.x, o.x), ey = fmaf(t, d.y, o.y), ez = fmaf(t, d.z, o.z);
    // (fminf and fmaxf skip the NaN of an unlimited ray with d = 0 along the axis)
    uint32_t m = 0;
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        if (!((sc.layer_axes >> a) & 1u)) continue;
        const float b = pick(a, o.x, o.y, o.z), e = pick(a, ex, ey, ez);
        const float l = fminf(b, e), h = fmaxf(b, e);
#pragma unroll
        for (int c = 0; c < kMaxClusters; ++c)   // unused entries are empty slabs
            m |= h >= sc.layer_lo[a][c] && l <= sc.layer_hi[a][c] ? 1u << c : 0u;
    }
    return m;
}

// A leaf's triangles are tested once fewer lanes than kRunMin walk and fewer
// than that descend (2e7 photons on the DARWIN-scale mesh: 92 ms with 8, 98
// with 4 or 12, at the time); a part of the traversal runs until half of the
// lanes that wanted it are through.
constexpr int kRunMin = 8;

// Lets the queries of a warp run until `need` of its n0 queries in flight have
// finished (node kDone).  q: the lane's slot.
template <bool kStats, class Lap>
__device__ __forceinline__ void run_queries(const Scene& sc, const float4* q, uint32_t skip, const RayInv& r, float eps,
                                            int n0, int need, Query& cur, int* stack, int* err, Counters& cnt, Lap&& lap)
{
    const uint32_t lane = threadIdx.x & 31u;
    int node = cur.node, sp = cur.sp, seen = cur.seen;
    float bt = cur.bt, tw = cur.tw;
    uint32_t rec = cur.rec;
    int leaf = 0;   // parked leaf (0 = none: reference 0 is an internal node, never a leaf)
    // Each pass runs the part of the traversal that most lanes wait
    // for: a leaf's triangles, a step of the walk, a node.  A lane
    // with a parked leaf walks or descends on until it meets the next.
    while (true) {
        if (leaf == 0 && is_leaf(node)) {
            leaf = node;
            node = stack[--sp];
        }
        if (node == kWalk && tw > bt) node = stack[--sp];
        const int nw = __popc(__ballot_sync(FULL_MASK, node == kWalk));
        const int nd = __popc(__ballot_sync(FULL_MASK, node >= 0));
        const int nl = __popc(__ballot_sync(FULL_MASK, leaf != 0));
        if (nl > 0 && nw < kRunMin && nd < kRunMin) {
            const int stop = nl / 2;
            do {
                if (kStats && lane == 0) cnt.leaf_iters++;
                if (leaf != 0) {
                    const float4 o = q[0], sh = q[4];   // origin and shear constants wait in the slot
                    triangle(sc, WRay{o.x, o.y, o.z, sh.x, sh.y, sh.z, cur.kz}, skip, leaf, bt, rec, err);
                    if (kStats) {
                        cnt.q_leaves += leaf == 0;
                        cnt.tris++;
                    }
                }
            } while (__popc(__ballot_sync(FULL_MASK, leaf != 0)) > stop);
            lap(cnt.cyc[kCycLeaf], n0);
        } else if (nw == 0 && nd == 0) {
            break;
        } else if (nw >= nd) {
            const int stop = nw / 2;
            do {
                if (kStats && lane == 0) cnt.walk_iters++;
                if (node == kWalk) {
                    if (kStats) cnt.walks++;
                    walk_step(sc, q, r, eps, bt, tw, node, seen, stack, sp, err);
                }
            } while (__popc(__ballot_sync(FULL_MASK, node == kWalk)) > stop);
            lap(cnt.cyc[kCycNode], n0);
        } else {
            const int stop = nd / 2;
            do {
                if (kStats && lane == 0) cnt.node_iters++;
                if (node >= 0) {
                    if (kStats) cnt.q_nodes++;
                    node_visit(sc, r, bt * kBoxSlack, node, stack, sp, err);
                }
            } while (__popc(__ballot_sync(FULL_MASK, node >= 0)) > stop);
            lap(cnt.cyc[kCycNode], n0);
        }
        if (n0 - __popc(__ballot_sync(FULL_MASK, node != kDone || leaf != 0)) >= need) break;
    }
    // a parked leaf goes back under the part of the query that is left
    if (leaf != 0) {
        stack[sp++] = node;
        node = leaf;
    }
    cur.node = node;
    cur.sp = sp;
    cur.seen = seen;
    cur.bt = bt;
    cur.tw = tw;
    cur.rec = rec;
}

// ---------------------------------------------------------------------------
// rays given by the caller
// ---------------------------------------------------------------------------
// Fewer rays than this: k_trace_few.  Time of k_trace_few over that of k_trace,
// rays without / with free-flight limits:
//                          1e5 rays      2e5           4e5           8e5
//   small TPC              0.82 / 0.90   1.14 / 1.17   1.37 / 1.39   1.59 / 1.61
//   50 cm TPC              1.13 / 0.92   1.29 / 1.19   1.44 / 1.47   1.64 / 1.77
//   3000 loose triangles   1.12 / 1.04   1.53 / 1.55   1.81 / 1.88   2.18 / 2.14
//   box of 16 triangles    0.52 / 0.56   0.81 / 0.80   1.00 / 0.95   1.19 / 1.20
//   DARWIN-scale mesh      0.80 / 0.81   0.89 / 0.88   0.96 / 0.98   1.06 / 1.26
//   the same, wires        0.68 / 0.73   0.80 / 0.75   0.97 / 0.92   1.09 / 1.16
// The line lies where the last of them break even, within 8 %.
constexpr uint32_t kTraceMany = 400000;
// Few rays: one lane a ray to its end through layers and main tree.  Little
// code, which is what counts when the kernel lasts as long as a few hundred
// instruction fetches (1000 rays in the small TPC: 18 us, with the kernel below
// 41); `width` rays a warp, so that the rays do not wait for one another.
__global__ void k_trace_few(const __grid_constant__ Scene sc, const float* __restrict__ org,
                            const float* __restrict__ dir, const uint32_t* __restrict__ skip,
                            const float* __restrict__ tmax, uint32_t n, int width, uint32_t* __restrict__ hit,
                            float* __restrict__ t, int* err)
{
    const uint64_t i = (uint64_t)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * width + (threadIdx.x & 31u);
    if ((int)(threadIdx.x & 31u) >= width || i >= n) return;
    const float3 o = f3(org[3 * i], org[3 * i + 1], org[3 * i + 2]);
    const float3 d = f3(dir[3 * i], dir[3 * i + 1], dir[3 * i + 2]);
    const uint32_t leave_out = skip ? skip[i] : LXO_NO_HIT;
    const WRay wr = wray_setup(o, d);
    const float3 from = near_origin(sc, o, d);
    const RayInv r = ray_inv(sc, from, d);
    int stack[kStackSize];
    Query c = begin_query(sc, from, d, wr.kz, tmax ? tmax[i] : INFINITY, (1u << sc.n_clusters) - 1u, -1.0f, stack);
    int leaf = 0;   // parked leaf
    // "while-while" with postponed leaves (Aila & Laine, HPG 2009): a lane
    // that reaches a leaf parks it and descends on until every lane has one
    while (true) {
        while (c.node >= 0) {
            node_visit(sc, r, c.bt * kBoxSlack, c.node, stack, c.sp, err);
            if (leaf == 0 && is_leaf(c.node)) {
                leaf = c.node;
                c.node = stack[--c.sp];
            }
            if (!__any_sync(__activemask(), leaf == 0)) break;
        }
        if (leaf == 0 && is_leaf(c.node)) {
            leaf = c.node;
            c.node = stack[--c.sp];
        }
        while (leaf != 0) {
            do triangle(sc, wr, leave_out, leaf, c.bt, c.rec, err); while (leaf != 0);
            if (is_leaf(c.node)) {
                leaf = c.node;
                c.node = stack[--c.sp];
            }
        }
        if (c.node == kDone) break;
    }
    hit[i] = c.rec == LXO_NO_HIT ? LXO_NO_HIT : __float_as_uint(__ldg(sc.tris + 3 * (size_t)c.rec + 2).y);
    t[i] = c.rec == LXO_NO_HIT ? INFINITY : c.bt;
}

// Many rays.  A warp looks at 32 rays at a time: those whose whole flight the empty cubes
// clear are answered at once, the others wait in a ring of the warp's own,
// from which its lanes take their next ray when half of those in flight have
// finished.  What bounds it is the wait for nodes and triangles (60 % of a
// warp's cycles; L1 hits 40 %, L2 52 %, DRAM 13 % in use), with 15.8 of 32 lanes
// at work, and the last rays (an SM is busy for some 80 % of the time).  2e6 rays
// with free-flight limits in the DARWIN-scale mesh: 240 us, 397 with a lane a
// ray to the end of the warp's slowest and whole trees searched.
constexpr int kTraceThreads = 128, kTraceCtas = 9, kTraceWarps = kTraceThreads / 32, kTraceRing = 64;

__global__ void __launch_bounds__(kTraceThreads, kTraceCtas)
    k_trace(const __grid_constant__ Scene sc, const float* __restrict__ org, const float* __restrict__ dir,
            const uint32_t* __restrict__ skip, const float* __restrict__ tmax, uint32_t n,
            uint32_t* __restrict__ hit, float* __restrict__ t, int* err)
{
    __shared__ float4 s_slot[kTraceThreads * kSlotF4];
    __shared__ uint2 s_ring[kTraceWarps][kTraceRing];   // ray, layers | clear part of its flight << 16 (1 / 64 cells)
    float4* q = s_slot + kSlotF4 * threadIdx.x;
    uint2* ring = s_ring[threadIdx.x >> 5];
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t stride = (uint64_t)gridDim.x * kTraceWarps * 32u;
    uint64_t next = ((uint64_t)blockIdx.x * kTraceWarps + (threadIdx.x >> 5)) * 32u;
    uint32_t head = 0, tail = 0;   // ring entries taken and put, warp-uniform
    uint32_t ray = 0;
    bool have = false;
    uint32_t leave_out = 0;        // triangle id not to be hit
    float eps = 0.0f;
    RayInv r{};
    Query cur{kDone, 1, 0, kDone, 0.0f, 0.0f, LXO_NO_HIT};
    int stack[kStackSize];
    Counters cnt{};
    auto lap = [](unsigned long long&, int) {};
    while (true) {
        const uint32_t idle = __ballot_sync(FULL_MASK, !have);
        while (next < n && tail - head < (uint32_t)__popc(idle)) {   // at most 31 + 32 entries
            const uint64_t i = next + lane;
            bool wait = false;
            uint32_t word = 0;
            if (i < n) {
                const float3 o = f3(org[3 * i], org[3 * i + 1], org[3 * i + 2]);
                const float3 d = f3(dir[3 * i], dir[3 * i + 1], dir[3 * i + 2]);
                const float tm = tmax ? tmax[i] : INFINITY;
                const RayInv ri = ray_inv(sc, o, d);
                // directions of any length: t of one cell along the main
                // axis; the main tree is searched where the numbers might not
                // carry the walk (0, infinite, NaN)
                const float cell = fminf(fminf(fabsf(ri.ix), fabsf(ri.iy)), fabsf(ri.iz));
                float clear_to = -1.0f;
                bool clear = false;
                if (cell > 1e-18f * sc.grid_h && cell < 1e18f * sc.grid_h)
                    clear = clear_flight(sc, o, d, tm, ri, 0.002f * cell, clear_to);
                const uint32_t layers = cluster_mask(sc, o, d, tm);
                wait = tm > 0.0f && !(clear && layers == 0u);
                if (!wait) {
                    hit[i] = LXO_NO_HIT;
                    t[i] = INFINITY;
                }
                word = layers | ((clear_to >= 0.0f ? min((uint32_t)__fdividef(64.0f * clear_to, cell), kNoWalk - 1u)
                                                   : kNoWalk) << 16);
            }
            const uint32_t m = __ballot_sync(FULL_MASK, wait);
            if (wait) ring[(tail + __popc(m & ((1u << lane) - 1u))) % kTraceRing] = make_uint2((uint32_t)i, word);
            tail += __popc(m);
            next += stride;
        }
        __syncwarp();
        const uint32_t take = min(tail - head, (uint32_t)__popc(idle));
        const uint32_t rank = __popc(idle & ((1u << lane) - 1u));
        if (((idle >> lane) & 1u) && rank < take) {
            const uint2 e = ring[(head + rank) % kTraceRing];
            ray = e.x;
            const float3 o = f3(org[3ull * ray], org[3ull * ray + 1], org[3ull * ray + 2]);
            const float3 d = f3(dir[3ull * ray], dir[3ull * ray + 1], dir[3ull * ray + 2]);
            leave_out = skip ? skip[ray] : LXO_NO_HIT;
            const uint32_t units = e.y >> 16;
            const float3 from = units == kNoWalk ? near_origin(sc, o, d) : o;
            r = ray_inv(sc, from, d);
            const float cell = fminf(fminf(fabsf(r.ix), fabsf(r.iy)), fabsf(r.iz));
            eps = 0.002f * cell;
            float3 sh;
            const int kz = shear(d, sh);
            q[0] = make_float4(o.x, o.y, o.z, 0.0f);
            q[1] = make_float4(d.x, d.y, d.z, 0.0f);
            q[4] = make_float4(sh.x, sh.y, sh.z, 0.0f);
            cur = begin_query(sc, from, d, kz, tmax ? tmax[ray] : INFINITY, e.y & 0xFFu,
                              units != kNoWalk ? (float)units * (cell * (1.0f / 64.0f)) : -1.0f, stack);
            have = true;
        }
        head += take;
        const int n0 = __popc(__ballot_sync(FULL_MASK, have));
        if (n0 == 0) break;   // then the ring is empty and no ray is left
        run_queries<false>(sc, q, leave_out, r, eps, n0, max(1, n0 / 2), cur, stack, err, cnt, lap);
        if (have && cur.node == kDone) {
            hit[ray] = cur.rec == LXO_NO_HIT ? LXO_NO_HIT : __float_as_uint(__ldg(sc.tris + 3 * (size_t)cur.rec + 2).y);
            t[ray] = cur.rec == LXO_NO_HIT ? INFINITY : cur.bt;
            have = false;
        }
    }
}

// ---------------------------------------------------------------------------
// photon source
// ---------------------------------------------------------------------------
struct Photon {
    float3 pos, dir, pol;
    float time;
    float wl;             // wavelength, nm (set only when some material has dispersion)
    int medium;
    uint32_t last;
    uint32_t step;
    uint64_t pid;
};

__device__ __forceinline__ float3 random_pol(float3 k, float u)
{
    float3 e1, e2;
    onb(k, e1, e2);
    float s, c;
    sincospif(2.0f * u, &s, &c);
    return normalize(c * e1 + s * e2);
}

// Inside the regular polygon?  The point was drawn at azimuth 2 pi u inside
// the circumscribed circle, so only the side of its angular sector can bound
// it (the polygon is the union of the triangles centre-side).
__device__ __forceinline__ bool inside_poly(const SourceDev& s, float x, float y, float u_azimuth)
{
    if (s.n_sides <= 0) return true;
    float t = u_azimuth - s.phase_turns;
    t -= floorf(t);
    const int k = min((int)(t * (float)s.n_sides), s.n_sides - 1);
    return x * s.side_cos[k] + y * s.side_sin[k] <= s.apothem;
}

// Emission delay of the scintillation time profile (Sec. 2.2, Table 2): a
// mixture of two exponentials, from its own draw of the source step.
__device__ __forceinline__ float emission_delay(const U4& u, const TimeProfile& tp)
{
    if (tp.tau_s == 0.0f && tp.tau_t == 0.0f) return 0.0f;
    const float tau = u.u0 < tp.f_s ? tp.tau_s : tp.tau_t;
    return -tau * logf(u.u1);
}

// Wavelength from the Gaussian emission spectrum (Sec. 2.2, Table 2): the
// Box-Muller transform of the last two uniforms of the emission draw.
__device__ __forceinline__ float emission_wavelength(const U4& u, const Spectrum& sp)
{
    if (sp.sigma == 0.0f) return sp.mean;
    float s, c;
    sincospif(2.0f * u.u3, &s, &c);
    return fmaf(sp.sigma, sqrtf(-2.0f * logf(u.u2)) * c, sp.mean);
}

// Index and slowness (n / c) of a material at the photon's wavelength: the
// table values unless some material has dispersion (the kSpectral build of
// the propagation kernel, whose photons carry a wavelength).
template <bool kSpectral>
__device__ __forceinline__ float n_at(const DevMaterial& m, float wl)
{
    return kSpectral ? fmaf(m.dn, wl - LXO_REF_WAVELENGTH_NM, m.n) : m.n;
}

template <bool kSpectral>
__device__ __forceinline__ float n_over_c_at(const DevMaterial& m, float wl)
{
    return kSpectral ? fmaf(m.dn_over_c, wl - LXO_REF_WAVELENGTH_NM, m.n_over_c) : m.n_over_c;
}

// The emission draw, if the time profile or the spectrum needs it.
template <int kRounds>
__device__ __forceinline__ U4 emission_draw(const PropParams& p, uint64_t pid, const TimeProfile& tp, const Spectrum& sp,
                                            bool want_wl)
{
    if (tp.tau_s == 0.0f && tp.tau_t == 0.0f && (!want_wl || sp.sigma == 0.0f)) return U4{0.5f, 0.5f, 0.5f, 0.5f};
    return draw4<kRounds>(p.seed, pid, kSourceStep, 0xFFFFFFFFu);
}

// Event of global photon index idx (binary search on the prefix sums) and
// the photon's first state: direction and polarisation as for any source,
// position from the event's point / segment / ball.
// kRounds: see philox4x32_10; want_wl: the wavelength is wanted.
template <int kRounds>
__device__ Photon make_event_photon(const PropParams& p, uint64_t idx, bool want_wl)
{
    uint32_t lo = 0, hi = p.n_events;  // find e with prefix[e] <= idx < prefix[e+1]
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(&p.ev_prefix[mid]) <= idx) lo = mid; else hi = mid;
    }
    const EventDev ev = p.events[lo];
    Photon ph;
    ph.pid = ((uint64_t)(p.first_event + lo) << 32) | (uint64_t)(idx - __ldg(&p.ev_prefix[lo]));
    ph.medium = ev.medium;
    const U4 em = emission_draw<kRounds>(p, ph.pid, ev.prof, ev.spec, want_wl);
    ph.time = ev.t0 + emission_delay(em, ev.prof);
    ph.wl = want_wl ? emission_wavelength(em, ev.spec) : 0.0f;
    ph.last = LXO_NO_HIT;
    ph.step = 0;
    const U4 u = draw4<kRounds>(p.seed, ph.pid, kSourceStep, 0);
    const float c = 2.0f * u.u0 - 1.0f, sn = sqrtf(fmaxf(0.0f, 1.0f - c * c));
    float sp, cp;
    sincospif(2.0f * u.u1, &sp, &cp);
    ph.dir = f3(sn * cp, sn * sp, c);
    ph.pol = random_pol(ph.dir, u.u2);
    if (ev.kind == LXO_SRC_SEGMENT) {
        ph.pos = f3(ev.center[0] + u.u3 * (ev.p1[0] - ev.center[0]), ev.center[1] + u.u3 * (ev.p1[1] - ev.center[1]),
                    ev.center[2] + u.u3 * (ev.p1[2] - ev.center[2]));
    } else {
        ph.pos = f3(ev.center[0], ev.center[1], ev.center[2]);
        if (ev.kind == LXO_SRC_BALL) {
#pragma unroll 1
            for (int tr = 0; tr < kMaxTries; ++tr) {
                const U4 w = draw4<kRounds>(p.seed, ph.pid, kSourceStep, 1 + tr);
                const float x = ev.radius * (2.0f * w.u0 - 1.0f), y = ev.radius * (2.0f * w.u1 - 1.0f),
                            z = ev.radius * (2.0f * w.u2 - 1.0f);
                if (x * x + y * y + z * z <= ev.radius * ev.radius) {
                    ph.pos = f3(ev.center[0] + x, ev.center[1] + y, ev.center[2] + z);
                    break;
                }
            }
        }
    }
    return ph;
}

template <int kRounds>
__device__ Photon make_photon(const PropParams& p, uint64_t idx, bool want_wl)
{
    if (p.n_events) return make_event_photon<kRounds>(p, idx, want_wl);
    const SourceDev& s = p.src;
    Photon ph;
    ph.pid = p.base + idx;
    ph.medium = s.medium;
    const U4 em = emission_draw<kRounds>(p, ph.pid, s.prof, s.spec, want_wl);
    ph.time = s.t0 + emission_delay(em, s.prof);
    ph.wl = want_wl ? emission_wavelength(em, s.spec) : 0.0f;
    ph.last = LXO_NO_HIT;
    ph.step = 0;
    if (s.kind == LXO_SRC_EXPLICIT) {
        ph.pos = f3(s.pos[3 * idx], s.pos[3 * idx + 1], s.pos[3 * idx + 2]);
        ph.dir = normalize(f3(s.dir[3 * idx], s.dir[3 * idx + 1], s.dir[3 * idx + 2]));
        float3 e = f3(s.pol[3 * idx], s.pol[3 * idx + 1], s.pol[3 * idx + 2]);
        ph.pol = normalize(e - dot(e, ph.dir) * ph.dir);
        return ph;
    }
    const U4 u = draw4<kRounds>(p.seed, ph.pid, kSourceStep, 0);
    const float c = 2.0f * u.u0 - 1.0f, sn = sqrtf(fmaxf(0.0f, 1.0f - c * c));
    float sp, cp;
    sincospif(2.0f * u.u1, &sp, &cp);
    ph.dir = f3(sn * cp, sn * sp, c);
    ph.pol = random_pol(ph.dir, u.u2);
    if (s.kind == LXO_SRC_POINT) {
        ph.pos = f3(s.center[0], s.center[1], s.center[2]);
    } else if (s.kind == LXO_SRC_SEGMENT) {
        ph.pos = f3(s.center[0] + u.u3 * (s.p1[0] - s.center[0]), s.center[1] + u.u3 * (s.p1[1] - s.center[1]),
                    s.center[2] + u.u3 * (s.p1[2] - s.center[2]));
    } else if (s.kind == LXO_SRC_BALL) {
        ph.pos = f3(s.center[0], s.center[1], s.center[2]);
#pragma unroll 1
        for (int tr = 0; tr < kMaxTries; ++tr) {
            const U4 w = draw4<kRounds>(p.seed, ph.pid, kSourceStep, 1 + tr);
            const float x = s.radius * (2.0f * w.u0 - 1.0f), y = s.radius * (2.0f * w.u1 - 1.0f),
                        z = s.radius * (2.0f * w.u2 - 1.0f);
            if (x * x + y * y + z * z <= s.radius * s.radius) {
                ph.pos = f3(s.center[0] + x, s.center[1] + y, s.center[2] + z);
                break;
            }
        }
    } else {
        ph.pos = f3(0.0f, 0.0f, s.z_min + u.u3 * (s.z_max - s.z_min));
#pragma unroll 1
        for (int tr = 0; tr < kMaxTries; ++tr) {
            const U4 w = draw4<kRounds>(p.seed, ph.pid, kSourceStep, 1 + tr);
            float r = s.radius * sqrtf(w.u0), sa, ca;
            sincospif(2.0f * w.u1, &sa, &ca);
            if (inside_poly(s, r * ca, r * sa, w.u1)) {
                ph.pos.x = r * ca;
                ph.pos.y = r * sa;
                break;
            }
            r = s.radius * sqrtf(w.u2);
            sincospif(2.0f * w.u3, &sa, &ca);
            if (inside_poly(s, r * ca, r * sa, w.u3)) {
                ph.pos.x = r * ca;
                ph.pos.y = r * sa;
                break;
            }
        }
    }
    return ph;
}

// 588 instructions a photon (three generator calls, six sines and cosines, two
// logarithms) would be 58 us for 4e6 photons at one a cycle and scheduler; it
// takes 84, with 69 % of the issue slots in use.  In the others no warp is ready:
// they wait for busy pipes (the one for indexed constants, the sides of the
// polygon, 64 %, integer 51 %) and for results of the special functions.  The
// stores are plain, since they are not what it waits for (LSU 6 % in use, DRAM
// 17 %): through shared memory, in full lines, the kernel took 98 us, with 90
// before the two emission draws became one and 84 now.
constexpr int kSampleThreads = 128;

__global__ void k_sample_source(const __grid_constant__ PropParams p, float* pos, float* dir, float* pol,
                                float* time, float* wavelength)
{
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.n) return;
    const Photon ph = make_photon<10>(p, i, wavelength != nullptr);
    pos[3 * i] = ph.pos.x; pos[3 * i + 1] = ph.pos.y; pos[3 * i + 2] = ph.pos.z;
    dir[3 * i] = ph.dir.x; dir[3 * i + 1] = ph.dir.y; dir[3 * i + 2] = ph.dir.z;
    pol[3 * i] = ph.pol.x; pol[3 * i + 1] = ph.pol.y; pol[3 * i + 2] = ph.pol.z;
    if (time) time[i] = ph.time;
    if (wavelength) wavelength[i] = ph.wl;
}

// ---------------------------------------------------------------------------
// interactions (Sec. 2.2; Appendix items 1 and 3)
// ---------------------------------------------------------------------------

// Rayleigh scattering, dipole law: density of the new direction k' is
// proportional to 1 - (k'.eps)^2; new polarisation = eps projected
// perpendicular to k'.  Sampled without a loop, in the frame whose pole is
// eps: c = cos(k', eps) from the inverse of its CDF, the cubic c^3 - 3c =
// 2 - 4 u0, c = 2 cos((acos(1 - 2 u0) + 4 pi) / 3); azimuth 2 pi u1 in
// onb(eps).  With w the unit azimuthal vector, k' = c eps + s w and the
// projection of eps perpendicular to k' is s (s eps - c w), s = sin.
__device__ __forceinline__ void rayleigh(Photon& ph, uint64_t seed)
{
    const U4 u = draw4(seed, ph.pid, ph.step, 1);
    const float a = acosf(1.0f - 2.0f * u.u0) * 0.318309886183790672f;   // in units of pi
    const float c = 2.0f * cospif((a + 4.0f) * (1.0f / 3.0f));
    const float s = sqrtf(fmaxf(0.0f, 1.0f - c * c));
    float sp, cp;
    sincospif(2.0f * u.u1, &sp, &cp);
    float3 e1, e2;
    onb(ph.pol, e1, e2);
    const float3 w = cp * e1 + sp * e2;
    const float3 eps = ph.pol;
    ph.dir = normalize(c * eps + s * w);
    ph.pol = normalize(s * eps - c * w);
}

// Lambertian reflection about the incident-side normal N (draw 1 of the step)
__device__ __forceinline__ void lambert(Photon& ph, float3 N, uint64_t seed)
{
    const U4 u = draw4(seed, ph.pid, ph.step, 1);
    const float c = sqrtf(u.u0), sn = sqrtf(fmaxf(0.0f, 1.0f - u.u0));
    float sp, cp;
    sincospif(2.0f * u.u1, &sp, &cp);
    float3 t1, t2;
    onb(N, t1, t2);
    ph.dir = normalize(c * N + sn * (cp * t1 + sp * t2));
    ph.pol = random_pol(ph.dir, u.u2);
}

__device__ __forceinline__ void mirror(Photon& ph, float3 N)
{
    const float ci = -dot(ph.dir, N);
    const float pe = dot(ph.pol, N);
    ph.dir = normalize(ph.dir + (2.0f * ci) * N);
    float3 e = (2.0f * pe) * N - ph.pol;
    e = e - dot(e, ph.dir) * ph.dir;
    ph.pol = normalize(e);
}

// Fresnel at a bare dielectric boundary n1 -> n2 with a linearly polarised
// photon: P(reflect) = cs^2 Rs + cp^2 Rp; outgoing polarisation is the
// coherent sum of the s and p amplitudes (p basis = s x k of each wave;
// magnitudes only under total internal reflection).  Normal incidence:
// s = eps (Appendix item 1).  Returns true if reflected.
__device__ __forceinline__ bool dielectric(Photon& ph, float3 N, float n1, float n2, float u)
{
    const float3 k = ph.dir;
    const float ci = fminf(1.0f, -dot(k, N));
    float3 s = cross(k, N);
    const float sl2 = dot(s, s);
    s = (sl2 < 1e-12f) ? ph.pol : rsqrtf(sl2) * s;
    const float3 pin = cross(s, k);
    const float cs = dot(ph.pol, s), cpv = dot(ph.pol, pin);
    const float eta = n1 / n2;
    const float st2 = eta * eta * (1.0f - ci * ci);
    float rs = 1.0f, rp = 1.0f, ts = 0.0f, tp = 0.0f, ct = 0.0f, pr = 1.0f;
    const bool tir = st2 >= 1.0f;
    if (!tir) {
        ct = sqrtf(1.0f - st2);
        const float a = n1 * ci, b = n2 * ct, c2 = n2 * ci, d2 = n1 * ct;
        // one fast reciprocal per denominator (2 ulp; the physics is float32
        // and statistical, unlike the exact intersection)
        const float i1 = __fdividef(1.0f, a + b), i2 = __fdividef(1.0f, c2 + d2);
        rs = (a - b) * i1;
        rp = (c2 - d2) * i2;
        ts = 2.0f * a * i1;
        tp = 2.0f * a * i2;
        pr = cs * cs * rs * rs + cpv * cpv * rp * rp;
    }
    if (u < pr) {
        const float3 kr = normalize(k + (2.0f * ci) * N);
        const float3 pr_v = cross(s, kr);
        const float as = tir ? cs : cs * rs, ap = tir ? cpv : cpv * rp;
        ph.dir = kr;
        ph.pol = normalize(as * s + ap * pr_v);
        return true;
    }
    const float3 kt = normalize(eta * k + (eta * ci - ct) * N);
    const float3 pt_v = cross(s, kt);
    ph.dir = kt;
    ph.pol = normalize((cs * ts) * s + (cpv * tp) * pt_v);
    return false;
}

__device__ __forceinline__ float fmax3(float a, float b, float c) { return fmaxf(a, fmaxf(b, c)); }

// move off the surface just hit by a margin above the rounding of the hit point
__device__ __forceinline__ void spawn_offset(Photon& ph, float3 o_ray, float t_hit, float3 N, float side)
{
    float m = fmaxf(fmaxf(1.0f, t_hit), fmaxf(fmax3(fabsf(ph.pos.x), fabsf(ph.pos.y), fabsf(ph.pos.z)),
                                              fmax3(fabsf(o_ray.x), fabsf(o_ray.y), fabsf(o_ray.z))));
    const float eps = m * 3.814697265625e-06f;  // 2^-18
    ph.pos = ph.pos + (side * eps) * N;
}

// First half of a step: the absorption / Rayleigh distances in the current
// medium (the first two uniforms of the step's draw).
struct StepDraw {
    float d_abs, d_ray;
};

template <bool kSpectral>
__device__ __forceinline__ StepDraw begin_step(const PropParams& p, const Photon& ph)
{
    const U4 u = draw4(p.seed, ph.pid, ph.step, 0);
    const DevMaterial& mt = p.mat[ph.medium];
    StepDraw sd;
    float ray_len = mt.ray_len;
    // (lambda / reference)^p as 2^(p log2(lambda / reference)), with the fast
    // base-2 logarithm (documented error: 2^-22 absolute on [0.5, 2], 2 ulp
    // elsewhere) in place of powf's exact-case handling
    if (kSpectral && mt.ray_exp != 0.0f)
        ray_len *= exp2f(mt.ray_exp * __log2f(ph.wl * (1.0f / LXO_REF_WAVELENGTH_NM)));
    // the accurate logarithm: the fast one's absolute error near u = 1 biases
    // the sampled distances by ~1e-4 mm, enough for the paired parity tests
    // of the adjoint tallies to see it (measured, 2 % faster)
    sd.d_abs = isinf(mt.abs_len) ? INFINITY : -mt.abs_len * logf(u.u0);
    sd.d_ray = isinf(ray_len) ? INFINITY : -ray_len * logf(u.u1);
    return sd;
}

// Second half of a step that met no surface: bulk absorption or Rayleigh
// scattering at the sampled distance d_int (absorbed: the absorption distance
// is the shorter one).  Returns -1 if the photon lives on, else its fate code
// (detail set to the material).
template <bool kAdjoint, bool kSpectral>
__device__ __forceinline__ int bulk_event(const PropParams& p, Photon& ph, float d_int, bool absorbed, int& detail,
                                          float* tl)
{
    if (isinf(d_int)) {
        detail = -1;
        return LXO_FATE_ESCAPED;
    }
    const DevMaterial& mt = p.mat[ph.medium];
    const int ms = kAdjoint ? p.adj_mat_slot[ph.medium] : -1;
    ph.pos = ph.pos + d_int * ph.dir;
    ph.time += d_int * n_over_c_at<kSpectral>(mt, ph.wl);
    if (kAdjoint && ms >= 0) tl[2 * ms] += d_int;
    if (absorbed) {
        detail = ph.medium;
        return LXO_FATE_BULK_ABS;
    }
    if (kAdjoint && ms >= 0) tl[2 * ms + 1] += 1.0f;
    rayleigh(ph, p.seed);
    ph.last = LXO_NO_HIT;
    return -1;
}

// Second half of a step that met triangle record `rec` at distance t: the
// interaction with its surface.  Returns -1 if the photon lives on, else its
// fate code (detail set to channel / surface / triangle).
template <bool kAdjoint, bool kSpectral>
__device__ __forceinline__ int surface_event(const PropParams& p, Photon& ph, float t, uint32_t rec, int& detail,
                                             float* tl)
{
    const DevMaterial& mt = p.mat[ph.medium];
    const int ms = kAdjoint ? p.adj_mat_slot[ph.medium] : -1;
    const float3 o_ray = ph.pos;
    ph.pos = ph.pos + t * ph.dir;
    ph.time += t * n_over_c_at<kSpectral>(mt, ph.wl);
    if (kAdjoint && ms >= 0) tl[2 * ms] += t;
    // geometric normal and attributes of the triangle hit (record in leaf order)
    if (LXO_CHECK_BOUNDS && rec >= p.sc.n_records) {
        atomicOr(p.err, kErrBounds);
        detail = -1;
        return LXO_FATE_GEOM_ERR;
    }
    const float4* tr = p.sc.tris + 3 * (size_t)rec;
    const float4 va = __ldg(tr + 0), vb = __ldg(tr + 1), vc = __ldg(tr + 2);
    const uint32_t id = __float_as_uint(vc.y);
    const uint2 at = make_uint2(__float_as_uint(vc.z), __float_as_uint(vc.w));
    // the step's first draw again (its first two uniforms gave the distances)
    const U4 u = draw4<1>(p.seed, ph.pid, ph.step, 0);
    const float3 e1 = f3(va.w - va.x, vb.x - va.y, vb.y - va.z);
    const float3 e2 = f3(vb.z - va.x, vb.w - va.y, vc.x - va.z);
    const float3 ng = normalize(cross(e1, e2));
    const bool forward = dot(ph.dir, ng) > 0.0f;
    const int mi = at.x & 0xFF, mo = (at.x >> 8) & 0xFF;
    const uint32_t sid = at.x >> 16;
    const int from = forward ? mi : mo, to = forward ? mo : mi;
    const float3 Nf = forward ? (-1.0f) * ng : ng;
    ph.last = id;
    if (sid == LXO_SURF_NONE) {
        if (from != ph.medium || to >= p.n_mat) {
            detail = (int)id;
            return LXO_FATE_GEOM_ERR;
        }
        const bool refl = dielectric(ph, Nf, n_at<kSpectral>(p.mat[from], ph.wl), n_at<kSpectral>(p.mat[to], ph.wl),
                                      u.u2);
        if (!refl) ph.medium = to;
        spawn_offset(ph, o_ray, t, Nf, refl ? 1.0f : -1.0f);
        return -1;
    }
    const DevSurface& sf = p.surf[sid];
    if (sf.type == LXO_SURF_ABSORBER) {
        detail = (int)sid;
        return LXO_FATE_SURF_ABS;
    }
    if (sf.type == LXO_SURF_PHOTOCATHODE) {
        const int ch = (int)at.y;
        if (ch < 0 || ch >= p.n_chan) {
            atomicOr(p.err, kErrChannel);
            detail = (int)id;
            return LXO_FATE_GEOM_ERR;
        }
        detail = ch;
        return (u.u2 < sf.qe) ? LXO_FATE_DETECTED : LXO_FATE_QE_FAIL;
    }
    bool specular;
    const int ss = kAdjoint ? p.adj_surf_slot[sid] : -1;
    const int base_k = 2 * p.adj_n_mats + 2 * ss;
    if (sf.type == LXO_SURF_REFLECTOR) {
        if (!(u.u2 < sf.R)) {
            detail = (int)sid;
            return LXO_FATE_SURF_ABS;
        }
        if (kAdjoint && ss >= 0) tl[base_k] += 1.0f;
        specular = u.u3 < sf.spec;
    } else if (sf.type == LXO_SURF_ELECTRODE_T) {
        if (u.u2 < sf.T) {
            if (from != ph.medium || to >= p.n_mat) {
                detail = (int)id;
                return LXO_FATE_GEOM_ERR;
            }
            if (kAdjoint && ss >= 0) tl[base_k] += 1.0f;
            ph.medium = to;
            spawn_offset(ph, o_ray, t, Nf, -1.0f);
            return -1;
        }
        if (!(u.u3 < sf.Rw)) {
            detail = (int)sid;
            return LXO_FATE_SURF_ABS;
        }
        if (kAdjoint && ss >= 0) tl[base_k + 1] += 1.0f;
        specular = draw4<1>(p.seed, ph.pid, ph.step, 1).u3 < sf.wspec;
    } else {
        detail = (int)id;
        return LXO_FATE_GEOM_ERR;
    }
    if (specular)
        mirror(ph, Nf);
    else
        lambert(ph, Nf, p.seed);
    spawn_offset(ph, o_ray, t, Nf, 1.0f);
    return -1;
}

// ---------------------------------------------------------------------------
// persistent propagation kernel
// ---------------------------------------------------------------------------
// A pool of photons per CTA.  Each photon lives in a slot in shared memory and
// waits there, between the parts of its steps, in one of five sets: ready (its
// next flight is to be traced), ready to enter a planar layer, bulk event due,
// surface event due, free (its fate to be tallied, a new photon to be made).
// A warp looks at the sets, takes up to 32 slots of one, does that work for
// them, and puts them into the sets of what comes next.  What bounds the loop
// is issue slots times lanes at work: the loop this replaced kept a photon in
// a lane for its whole life and ran every kind of work for the few lanes that
// needed it (9.3 lanes of 32 per instruction, 210 instructions per photon
// step of a warp; here 17.6 and 115).  The draws of the next step and its
// flight's set-up belong to the batch that ends the step before, with all
// lanes at work.
// Flights that meet nothing need no query: the walk grid's empty cubes clear
// them (over half of the DARWIN-scale mesh's steps), which pays only because
// the lanes of the others are then filled with other photons.
// Instruction fetch is what is left: the requests that miss the SM's
// instruction cache came at the same 0.515 per cycle and GPC in three versions
// of this loop, so hot code is kept short (82 KB -> 75 KB: 8 to 12 % less
// time).  So does the length of each warp's own chain: 20 instructions more in
// the choice of the next batch cost 3 to 7 %.
// Launch shape: CTAs of kPoolThreads threads, kPoolCtas per SM: 18 warps of 56
// registers each; 2e7 photons on the DARWIN-scale mesh / 3e6 on the 50 cm TPC
// took 63.1 / 11.4 ms, with 2 x 640 threads of 48 registers 66.5 / 12.0, with
// 2 x 512 of 64 66.8 / 11.4, with 3 x 384 of 56 66.4 / 11.4.
// Measured (1e8 photons on the DARWIN-scale mesh / 3e6 on the 50 cm TPC with
// dispersion / 2e6 on the mesh without electrodes, GB300): 503 / 21.0 / 17.7
// ms for the loop before, 305 / 11.5 / 10.0 ms now.
constexpr int kPoolThreads = 576, kPoolCtas = 2;
// A batch starts with the lanes of this many columns or more (24: 5 % slower,
// 30: 2 %); a warp leaves the traversal once half of its queries have finished
// (a third: 1 % slower).
constexpr int kBatchMin = 28;
// The last photons of a CTA are shared out: a batch takes at most 1 / kSpread of
// them, so that a photon's step does not wait for those of all others (3e5
// photons of the mesh without electrodes: 3.39 ms with 8, 3.61 with 18, the
// warps of the CTA, 4.29 with 30; 3e5 of the 50 cm TPC 2.70 / 2.87 / 3.29).
constexpr int kSpread = 8;
constexpr int kMaxSlots = 1024;       // 32 columns of 32
// a warp that has found nothing so often leaves (it holds no photon; the
// others go on with theirs)
constexpr uint32_t kPollLimit = 1u << 20;

// Where a slot's photon waits.
enum { kReady = 0, kReadyLayer, kBulk, kSurf, kFree, kSets };

// A set of slots: bit j of word l stands for slot 32 j + l, so that lane l of
// any warp takes slots of column l only, from its own word: no talk between
// the lanes, no bank conflicts on the words or the slots (12 instructions;
// packing the members of a set into the lanes by a prefix sum took 136 to
// 194).  A slot leaves by atomicAnd, so none is taken twice and nothing waits.
// `turn`: words are tried from that bit on, another for each warp.
__device__ __forceinline__ int claim(uint32_t* set, uint32_t lanes, int turn, uint32_t lane)
{
    int slot = -1;
    if ((lanes >> lane) & 1u) {
        const uint32_t w = *(volatile uint32_t*)&set[lane];
        if (w) {
            const uint32_t r = __funnelshift_r(w, w, turn);
            const int j = (__ffs(r) - 1 + turn) & 31;
            if ((atomicAnd(&set[lane], ~(1u << j)) >> j) & 1u) slot = 32 * j + (int)lane;
        }
    }
    __threadfence_block();   // a slot's contents are read after its bit was taken
    return slot;
}

// At most n of the lanes in `lanes`.
__device__ __forceinline__ uint32_t at_most(uint32_t lanes, int n)
{
    for (int m = __popc(lanes); m > n; --m) lanes &= lanes - 1u;
    return lanes;
}

__device__ __forceinline__ void put(uint32_t* set, int slot) { atomicOr(&set[slot & 31], 1u << (slot >> 5)); }

// Tally of one photon's fate: shared-memory fate counters, global per-channel
// counts and arrival-time histogram, optional per-photon record and adjoint
// sums.  Plain per-lane atomics: aggregating them over the lanes of a warp
// that hit the same counter (match + reduce) measured 3.8 % slower on the
// DARWIN-scale workload, where two lanes rarely tally the same channel at
// once.
template <bool kAdjoint>
__device__ __forceinline__ void tally(const PropParams& p, unsigned long long* s_f, const Photon& ph, int fate,
                                      int detail, const float* tl)
{
    // row of the per-channel tallies: the channel, or (event - first event) * P + channel for batched events
    const size_t row = p.n_events ? (size_t)((uint32_t)(ph.pid >> 32) - p.first_event) * p.n_chan + detail
                                  : (size_t)detail;
    if (LXO_CHECK_BOUNDS && (fate == LXO_FATE_DETECTED || fate == LXO_FATE_QE_FAIL) &&
        (detail < 0 || row >= (size_t)(p.n_events ? p.n_events : 1) * p.n_chan)) {
        atomicOr(p.err, kErrBounds);
        return;
    }
    if (kAdjoint && fate == LXO_FATE_DETECTED)
        for (int k = 0; k < p.adj_k; ++k) atomicAdd(&p.out.adjoint[row * p.adj_k + k], (double)tl[k]);
    atomicAdd(&s_f[fate], 1ull);
    atomicAdd(&s_f[7], (unsigned long long)ph.step);
    if (fate == LXO_FATE_BULK_ABS) atomicAdd(&s_f[LXO_FATES_FIXED + detail], 1ull);
    if (fate == LXO_FATE_SURF_ABS) atomicAdd(&s_f[LXO_FATES_FIXED + p.n_mat + detail], 1ull);
    if (fate == LXO_FATE_DETECTED || fate == LXO_FATE_QE_FAIL) {
        atomicAdd(&p.out.lce[row], 1u);
        if (fate == LXO_FATE_DETECTED) {
            atomicAdd(&p.out.det[row], 1u);
            if (p.out.hist) {
                const float b = floorf(ph.time / p.tbin);
                const uint32_t bin = (b >= (float)p.n_tbins || !(b >= 0.0f)) ? p.n_tbins : (uint32_t)b;
                atomicAdd(&p.out.hist[row * (p.n_tbins + 1) + bin], 1u);
            }
        }
    }
    const uint64_t idx = ph.pid - p.base;
    if (p.out.ph_fate) p.out.ph_fate[idx] = (uint32_t)fate;
    if (p.out.ph_detail) p.out.ph_detail[idx] = detail;
    if (p.out.ph_steps) p.out.ph_steps[idx] = ph.step;
    if (p.out.ph_time) p.out.ph_time[idx] = ph.time;
    if (p.out.ph_state) {
        float* o = p.out.ph_state + 9 * idx;
        o[0] = ph.pos.x; o[1] = ph.pos.y; o[2] = ph.pos.z;
        o[3] = ph.dir.x; o[4] = ph.dir.y; o[5] = ph.dir.z;
        o[6] = ph.pol.x; o[7] = ph.pol.y; o[8] = ph.pol.z;
    }
}

// Counting build: histogram of a step's node visits (8-wide bins) by medium
// (0 or another), and its leaves.
__device__ __forceinline__ void step_histogram(const PropParams& p, int medium, uint32_t dn, uint32_t dl)
{
    const int m = medium == 0 ? 0 : 1;
    atomicAdd(&p.out.stats[9 + 10 * m + min(dn / 8u, 8u)], 1ull);
    atomicAdd(&p.out.stats[9 + 10 * m + 9], (unsigned long long)dl);
}

// A slot: five float4.
//   [0] position, flight length (sign bit: absorption at its end) or hit distance
//   [1] direction, a word: ready: axis kz | cluster mask << 2 | clear units << 16;  after the
//       query: record hit (LXO_NO_HIT none);  free: fate (-1: no photon yet)
//   [2] polarisation, time
//   [3] id low, id high, step, medium << 28 | triangle left last
//   [4] the watertight test's shear constants, wavelength
__device__ __forceinline__ Photon load_slot(const float4* q)
{
    const float4 a = q[0], b = q[1], c = q[2], d = q[3];
    Photon ph;
    ph.pos = f3(a.x, a.y, a.z);
    ph.dir = f3(b.x, b.y, b.z);
    ph.pol = f3(c.x, c.y, c.z);
    ph.time = c.w;
    ph.wl = q[4].w;
    ph.pid = (uint64_t)__float_as_uint(d.x) | ((uint64_t)__float_as_uint(d.y) << 32);
    ph.step = __float_as_uint(d.z);
    const uint32_t lm = __float_as_uint(d.w);
    ph.medium = (int)(lm >> 28);
    ph.last = (lm & kNoTri) == kNoTri ? LXO_NO_HIT : (lm & kNoTri);
    return ph;
}

template <bool kStats, bool kAdjoint, bool kSpectral>
__global__ void __launch_bounds__(kPoolThreads, kPoolCtas) k_propagate(const __grid_constant__ PropParams p)
{
    extern __shared__ float4 s_pool[];   // [p.slots] slots, then the adjoint tallies [p.slots][p.tally_stride]
    __shared__ unsigned long long s_f[kMaxFates];
    __shared__ uint32_t s_set[kSets][32];
    __shared__ int s_live, s_dry;
    for (int i = threadIdx.x; i < p.n_fates; i += blockDim.x) s_f[i] = 0ull;
    for (int i = threadIdx.x; i < kSets * 32; i += blockDim.x) {
        const int rows = (p.slots - (i & 31) + 31) >> 5;   // slots of this column
        s_set[i >> 5][i & 31] = (i >> 5) != kFree || rows <= 0 ? 0u : (rows >= 32 ? FULL_MASK : (1u << rows) - 1u);
    }
    for (int i = threadIdx.x; i < p.slots; i += blockDim.x) s_pool[kSlotF4 * i + 1].w = __int_as_float(-1);
    if (threadIdx.x == 0) {
        s_live = p.slots;
        s_dry = 0;
    }
    __syncthreads();

    float* s_tally = reinterpret_cast<float*>(s_pool + kSlotF4 * p.slots);
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int warp = threadIdx.x >> 5;
    const int turn = warp & 31;
    // the lane's query in flight: its slot (-1 none) and state; its stack in local memory
    int slot = -1;
    Query cur{kDone, 1, 0, kDone, 0.0f, 0.0f, LXO_NO_HIT};
    int stack[kStackSize];
    uint32_t polls = 0;
    Counters cnt{};
    long long tick = kStats ? clock64() : 0;
    // counting build: adds the warp's cycles since the last call, times the lanes at work
    auto lap = [&](unsigned long long& sum, int lanes) {
        if (!kStats) return;
        const long long now = clock64();
        if (lane == 0) {
            sum += (unsigned long long)((now - tick) * lanes);
            cnt.loop_cycles += (unsigned long long)((now - tick) * lanes);
        }
        tick = now;
    };

    while (true) {
        uint32_t in[kSets];   // the lanes for which each set has a slot
#pragma unroll
        for (int k = 0; k < kSets; ++k) in[k] = __ballot_sync(FULL_MASK, *(volatile uint32_t*)&s_set[k][lane] != 0u);
        const int live = __shfl_sync(FULL_MASK, *(volatile int*)&s_live, 0);
        const uint32_t busy = __ballot_sync(FULL_MASK, slot >= 0);
        // a batch: 32 lanes, fewer once few photons are left
        const int width = min(32, (live + kSpread - 1) / kSpread);
        const int full = width > kBatchMin ? kBatchMin : max(width, 1);
        int stage;
        if (__popc(in[kBulk]) >= full) stage = kBulk;
        else if (__popc(in[kSurf]) >= full) stage = kSurf;
        else if (__popc(in[kFree]) >= full) stage = kFree;
        else if ((in[kReady] | in[kReadyLayer] | busy) != 0u) stage = kReady;
        else if (in[kBulk]) stage = kBulk;
        else if (in[kSurf]) stage = kSurf;
        else if (in[kFree]) stage = kFree;
        else {
            // nothing to do here: other warps hold the photons left
            if (live <= 0 || ++polls > kPollLimit) break;
            // (short sleeps take issue slots from the warps that work: 2e4
            // photons of the 50 cm TPC took 1.69 ms with 100 ns, 1.48 with 2 us)
            __nanosleep(2000);
            lap(cnt.idle_cycles, 32);
            continue;
        }

        if (stage == kReady) {
            // ---- traversal ------------------------------------------------
            bool fresh = false;
            const int room = width - __popc(busy);
            if (room > 0) {
                // queries that enter a layer's cells are taken apart from the others
                const uint32_t fr = in[kReady] & ~busy, fl = in[kReadyLayer] & ~busy;
                const int from = __popc(fl) > __popc(fr) ? kReadyLayer : kReady;
                const uint32_t f = from == kReady ? fr : fl;
                if (f) {
                    const int t = claim(s_set[from], room < 32 ? at_most(f, room) : f, turn, lane);
                    if (t >= 0) {
                        slot = t;
                        fresh = true;
                    }
                }
            }
            const int n0 = __popc(__ballot_sync(FULL_MASK, slot >= 0));
            if (n0 == 0) continue;
            const float4* q = s_pool + kSlotF4 * max(slot, 0);
            RayInv ray{};
            if (slot >= 0) {
                const float4 a = q[0], b = q[1];
                const float3 o = f3(a.x, a.y, a.z), d = f3(b.x, b.y, b.z);
                ray = ray_inv(p.sc, o, d);
                if (fresh) {
                    const uint32_t kw = __float_as_uint(b.w), units = kw >> 16;
                    cur = begin_query(p.sc, o, d, (int)(kw & 3u), fabsf(a.w), (kw >> 2) & 0xFFu,
                                      units != kNoWalk ? (float)units * p.sc.walk_unit : -1.0f, stack);
                }
            }
            __syncwarp();
            lap(cnt.cyc[kCycBegin], n0);
            if (kStats && lane == 0) cnt.entries++;
            const int need = max(1, n0 / 2);
            const uint32_t skip = __float_as_uint(q[3].w) & kNoTri;
            run_queries<kStats>(p.sc, q, skip, ray, p.sc.walk_eps, n0, need, cur, stack, p.err, cnt, lap);
            const bool done = slot >= 0 && cur.node == kDone;
            if (done) {
                float4* w = s_pool + kSlotF4 * slot;
                if (cur.rec != LXO_NO_HIT) w[0].w = cur.bt;
                w[1].w = __uint_as_float(cur.rec);
            }
            if (kStats && done) {
                step_histogram(p, (int)(__float_as_uint(q[3].w) >> 28), cnt.q_nodes, cnt.q_leaves);
                cnt.nodes += cnt.q_nodes;
                cnt.leaves += cnt.q_leaves;
                cnt.q_nodes = cnt.q_leaves = 0;
            }
            __threadfence_block();
            if (done) {
                put(s_set[cur.rec != LXO_NO_HIT ? kSurf : kBulk], slot);
                slot = -1;
            }
            __syncwarp();
            lap(cnt.cyc[kCycBegin], n0);
            continue;
        }

        // ---- interactions, tallies and new photons ------------------------
        const int want = stage == kFree ? min(width, (int)min(p.chunk, 32u)) : width;
        const uint32_t lanes = stage == kBulk ? in[kBulk] : (stage == kSurf ? in[kSurf] : in[kFree]);
        const int s = claim(s_set[stage], want < 32 ? at_most(lanes, max(want, 1)) : lanes, turn, lane);
        const uint32_t members = __ballot_sync(FULL_MASK, s >= 0);
        const int got = __popc(members);
        if (got == 0) continue;
        float4* q = s_pool + kSlotF4 * max(s, 0);
        float* tl = kAdjoint ? s_tally + (size_t)max(s, 0) * p.tally_stride : nullptr;
        Photon ph;
        bool alive = false;
        int fate = -1, detail = -1;
        if (s >= 0) ph = load_slot(q);
        if (stage == kFree) {
            if (s >= 0) {
                const int f = __float_as_int(q[1].w);
                if (f >= 0) tally<kAdjoint>(p, s_f, ph, f, __float_as_int(q[0].w), tl);
            }
            unsigned long long base = p.n;
            if (lane == 0 && !*(volatile int*)&s_dry) base = atomicAdd(p.queue, (unsigned long long)got);
            base = __shfl_sync(FULL_MASK, base, 0);
            const int avail = base < p.n ? (int)min((unsigned long long)got, (unsigned long long)p.n - base) : 0;
            if (lane == 0 && avail < got) {
                s_dry = 1;
                atomicSub(&s_live, got - avail);
            }
            const int rank = __popc(members & lt_mask);
            if (s >= 0 && rank < avail) {
                ph = make_photon<1>(p, base + rank, p.spectral != 0);
                if (kAdjoint)
                    for (int k = 0; k < p.adj_k; ++k) tl[k] = 0.0f;
                alive = true;
            }
        } else if (s >= 0) {
            const float4 a = q[0], b = q[1];
            if (stage == kBulk)
                fate = bulk_event<kAdjoint, kSpectral>(p, ph, fabsf(a.w), (__float_as_uint(a.w) >> 31) != 0u, detail, tl);
            else
                fate = surface_event<kAdjoint, kSpectral>(p, ph, a.w, __float_as_uint(b.w), detail, tl);
            ph.step++;
            if (fate < 0 && ph.step >= p.max_steps) {
                fate = LXO_FATE_TRUNCATED;
                detail = -1;
            }
            alive = fate < 0;
        }
        if (kStats) {
            if (lane == 0 && stage != kFree) {
                cnt.steps += got;
                cnt.batches++;
            }
            __syncwarp();
            lap(cnt.cyc[stage == kFree ? kCycRefill : kCycFinish], got);
        }
        int to = -1;
        if (alive) {
            // the next step's draws and its flight: clear of every triangle
            // by the table, or a query
            const StepDraw sd = begin_step<kSpectral>(p, ph);
            const float d = fminf(sd.d_abs, sd.d_ray);
            uint32_t word = LXO_NO_HIT;
            float3 sh = f3(0.0f, 0.0f, 0.0f);
            float clear_to;
            const uint32_t clusters = cluster_mask(p.sc, ph.pos, ph.dir, d);
            const bool clear = clear_flight(p.sc, ph.pos, ph.dir, d, ray_inv(p.sc, ph.pos, ph.dir), p.sc.walk_eps, clear_to);
            if (clear && clusters == 0u) {
                to = kBulk;
                if (kStats) step_histogram(p, ph.medium, 0, 0);
            } else {
                to = clusters ? kReadyLayer : kReady;
                const int k = shear(ph.dir, sh);
                const uint32_t units = clear_to >= 0.0f ? min((uint32_t)(clear_to * p.sc.walk_per_mm), kNoWalk - 1u) : kNoWalk;
                word = (uint32_t)k | (clusters << 2) | (units << 16);
            }
            const uint32_t ab = sd.d_abs <= sd.d_ray ? 0x80000000u : 0u;
            q[0] = make_float4(ph.pos.x, ph.pos.y, ph.pos.z, __uint_as_float(__float_as_uint(d) | ab));
            q[1] = make_float4(ph.dir.x, ph.dir.y, ph.dir.z, __uint_as_float(word));
            q[4] = make_float4(sh.x, sh.y, sh.z, ph.wl);
        } else if (fate >= 0) {
            to = kFree;
            q[0] = make_float4(ph.pos.x, ph.pos.y, ph.pos.z, __int_as_float(detail));
            q[1] = make_float4(ph.dir.x, ph.dir.y, ph.dir.z, __int_as_float(fate));
        }
        if (to >= 0) {
            q[2] = make_float4(ph.pol.x, ph.pol.y, ph.pol.z, ph.time);
            q[3] = make_float4(__uint_as_float((uint32_t)ph.pid), __uint_as_float((uint32_t)(ph.pid >> 32)),
                               __uint_as_float(ph.step),
                               __uint_as_float(((uint32_t)ph.medium << 28) | (ph.last & kNoTri)));
        }
        __threadfence_block();
        if (to >= 0) put(s_set[to], s);
        __syncwarp();
        lap(cnt.cyc[kCycDraw], got);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < p.n_fates; i += blockDim.x)
        if (s_f[i]) atomicAdd(&p.out.fates[i], s_f[i]);
    if (kStats) {
        unsigned long long* o = p.out.stats;
        atomicAdd(&o[0], (unsigned long long)cnt.steps);
        atomicAdd(&o[1], (unsigned long long)cnt.nodes);
        atomicAdd(&o[2], (unsigned long long)cnt.leaves);
        atomicAdd(&o[3], (unsigned long long)cnt.tris);
        atomicAdd(&o[4], (unsigned long long)cnt.node_iters);
        atomicAdd(&o[5], (unsigned long long)cnt.leaf_iters);
        atomicAdd(&o[6], (unsigned long long)cnt.batches);
        atomicAdd(&o[7], cnt.cyc[kCycNode] + cnt.cyc[kCycLeaf] + cnt.cyc[kCycBegin]);
        atomicAdd(&o[8], cnt.loop_cycles);
        for (int k = 0; k < kCycPhases; ++k) atomicAdd(&o[29 + k], cnt.cyc[k]);
        atomicAdd(&o[35], (unsigned long long)cnt.entries);
        atomicAdd(&o[36], cnt.idle_cycles);
        atomicAdd(&o[37], (unsigned long long)cnt.walks);
        atomicAdd(&o[38], (unsigned long long)cnt.walk_iters);
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_trace(const Scene& sc, const float* org, const float* dir, const uint32_t* skip,
                         const float* tmax, uint32_t n, uint32_t* hit, float* t, int* err, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (n < kTraceMany) {
        const uint64_t warps = (uint64_t)sms * 16u;
        const int width = (int)std::min<uint64_t>(32u, (n + warps - 1) / warps);
        const unsigned blocks = (unsigned)(((n + width - 1u) / width + kTraceWarps - 1) / kTraceWarps);
        k_trace_few<<<blocks, kTraceThreads, 0, st>>>(sc, org, dir, skip, tmax, n, width, hit, t, err);
        return cudaGetLastError();
    }
    k_trace<<<(unsigned)(sms * kTraceCtas), kTraceThreads, 0, st>>>(sc, org, dir, skip, tmax, n, hit, t, err);
    return cudaGetLastError();
}

cudaError_t launch_sample_source(const PropParams& p, float* pos, float* dir, float* pol, float* time,
                                 float* wavelength, cudaStream_t st)
{
    if (p.n == 0) return cudaSuccess;
    const uint64_t blocks = (p.n + kSampleThreads - 1) / kSampleThreads;
    k_sample_source<<<(unsigned)blocks, kSampleThreads, 0, st>>>(p, pos, dir, pol, time, wavelength);
    return cudaGetLastError();
}

cudaError_t launch_propagate(const PropParams& params, int device, cudaStream_t st)
{
    if (params.n == 0) return cudaSuccess;
    PropParams p = params;
    const bool stats = (p.flags & LXO_FLAG_STATS) != 0;
    const bool adj = (p.flags & LXO_FLAG_ADJOINT) != 0;
    auto kern = p.spectral ? (adj ? k_propagate<false, true, true> : k_propagate<false, false, true>)
                           : (adj ? k_propagate<false, true, false> : k_propagate<false, false, false>);
    if (stats)
        kern = p.spectral ? (adj ? k_propagate<true, true, true> : k_propagate<true, false, true>)
                          : (adj ? k_propagate<true, true, false> : k_propagate<true, false, false>);
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    // slots per CTA: what kPoolCtas CTAs leave of the SM's shared memory (164
    // KiB of it for the forward builds, all of it with the adjoint tallies)
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    p.tally_stride = adj ? (p.adj_k | 1) : 0;
    const size_t per_slot = sizeof(float4) * kSlotF4 + sizeof(float) * p.tally_stride;
    const size_t room = (size_t)(adj ? 227 : kPoolKb) * 1024 / kPoolCtas - 1024 - fa.sharedSizeBytes;
    const uint64_t slots = std::min<uint64_t>(kMaxSlots, room / per_slot / 32 * 32);
    // the kernel's limit is one value for all threads of the process: the room,
    // which does not depend on this launch's tallies
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPoolThreads, slots * per_slot);
    if (e != cudaSuccess) return e;
    // a launch shape set by the caller limits the threads per SM
    if (p.blocks_per_sm > 0)
        per_sm = std::min(per_sm, (int)((p.blocks_per_sm * p.block_threads + kPoolThreads - 1) / kPoolThreads));
    per_sm = std::max(1, per_sm);
    uint64_t blocks = std::min<uint64_t>((uint64_t)sms * per_sm, p.n);
    p.slots = (int)std::min<uint64_t>(slots, (p.n + blocks - 1) / blocks);
    kern<<<(unsigned)blocks, kPoolThreads, slots * per_slot, st>>>(p);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// adjoint backward: J[c][q] = a_q * sums[c][ia_q] + b_q * sums[c][ib_q];
// optional grad[q] = sum_c g[c] J[c][q]
// ---------------------------------------------------------------------------
struct AdjCoefs {
    AdjCoef c[2 * LXO_ADJ_MAX_MATERIALS + LXO_ADJ_MAX_SURFACES];
};

__global__ void k_adjoint_jacobian(const AdjCoefs co, int Q, int K, int P, const double* __restrict__ sums,
                                   double* __restrict__ J)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P * Q) return;
    const int ch = i / Q, q = i % Q;
    const AdjCoef& c = co.c[q];
    J[i] = c.a * sums[(size_t)ch * K + c.ia] + c.b * sums[(size_t)ch * K + c.ib];
}

__global__ void k_adjoint_vjp(int Q, int P, const double* __restrict__ J, const double* __restrict__ g,
                              double* __restrict__ grad)
{
    __shared__ double red[256];
    const int q = blockIdx.x;
    double acc = 0.0;
    for (int ch = threadIdx.x; ch < P; ch += blockDim.x) acc += g[ch] * J[(size_t)ch * Q + q];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) grad[q] = red[0];
}

cudaError_t launch_adjoint_jacobian(const AdjCoef* coef_host, int Q, int K, int P, const double* sums, double* J,
                                    const double* g, double* grad, cudaStream_t st)
{
    AdjCoefs co;
    for (int q = 0; q < Q; ++q) co.c[q] = coef_host[q];
    const int n = P * Q, threads = 256;
    k_adjoint_jacobian<<<(n + threads - 1) / threads, threads, 0, st>>>(co, Q, K, P, sums, J);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !g) return e;
    k_adjoint_vjp<<<Q, 256, 0, st>>>(Q, P, J, g, grad);
    return cudaGetLastError();
}

}  // namespace lxo
