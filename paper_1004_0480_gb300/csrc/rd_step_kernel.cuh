// rd_step_kernel.cuh -- the fused forward-Euler step kernels (sm_103a).
//
// The kernels share the per-cell update functions below, so every launch
// shape gives the same bits: rd_step_kernel (T steps per launch, any tile
// height, described here), rd_march_kernel (one or two steps per launch, even
// heights, models without Cahn-Hilliard), rd_step1w_kernel (one step, 8 cells
// per thread) and rd_marchch_kernel (one step, the Cahn-Hilliard models); the
// others are described where they are defined.
//
// rd_step_kernel: one launch advances T steps of eq. (5) for every species
// of every work item.  A work item is an x-y tile of 64 x TY cells and a chunk of z planes
// of one instance.  The CTA marches up the chunk, as the paper's Shared
// method does (Section 4.1, Table 4), restated for this hardware:
//
//  * thread layout: one thread per 4-cell vector position of the tile
//    widened by a halo (one vector each side in x, L rows each side in y),
//    i.e. (16 + 2) x (TY + 2L) threads.  As in the paper's overlapped
//    blocks, halo threads load (and at inner levels compute) but never
//    store.  A thread keeps its position for the whole march, so all index
//    and boundary arithmetic is done once per work item.
//  * level 0: planes of the current state arrive in a shared-memory ring by
//    per-thread cp.async copies, several planes ahead.
//  * level l = 1..L: as soon as level l-1 has planes q-1, q, q+1, plane q of
//    level l is computed from them; every level keeps a few planes in shared
//    memory.  Level L goes to global memory.  All levels advance once per
//    plane, with a single barrier per plane.
//  * Without Cahn-Hilliard L = T and level l is the state after l steps.
//    With it L = 2T: odd levels hold mu = f'(c) - kappa Lap c, even levels
//    the state -- the paper's "Laplacian, boundary rule, Laplacian"
//    biharmonic (Section 4.1), fused into the march.
//
// Boundary rules, applied at every level:
//   periodic axis  halo cells are real cells at wrapped coordinates;
//   zero flux      a neighbour outside the domain is the cell itself (the
//                  ghost equals the face cell), so outside cells are never
//                  read or loaded;
//   held layer     (Dirichlet) the cell's new value is its bc value.
// Every value at every level comes from the same per-cell update with
// explicitly rounded operations, and inner levels are rounded to the storage
// type, so a T-step launch reproduces T one-step launches bit for bit.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "rd_debug.cuh"
#include "rd_internal.h"
#include "rd_pack.cuh"

namespace rdk {

constexpr int kNQ = kTileQ + 2;       // vector positions per row incl. halo
constexpr int kRW = kNQ * kVEC;       // elements per shared-memory row

// ---------------------------------------------------------------- storage
template <class ST> struct Store;

// Loads and stores of 4-cell vectors and single cells in either space, and
// asynchronous global-to-shared copies.  In the bounds-checked debug build
// (rd_debug.cuh) each checks its shared-memory side and skips an access out
// of range (a load then yields 0); global sides are checked by the callers,
// which know the instance.
template <> struct Store<float> {
    __device__ __forceinline__ static void load(const float* p, float (&v)[4]) {
        if (!RD_DBG_ANY(p, 16, kSiteSharedLoad)) { v[0] = v[1] = v[2] = v[3] = 0.0f; return; }
        const float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    }
    __device__ __forceinline__ static void store(float* p, const float (&v)[4]) {
        if (!RD_DBG_ANY(p, 16, kSiteSharedStore)) return;
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
    __device__ __forceinline__ static float get(const float* p) {
        if (!RD_DBG_ANY(p, 4, kSiteSharedLoad)) return 0.0f;
        return *p;
    }
    __device__ __forceinline__ static float round(float x) { return x; }
    __device__ __forceinline__ static void cp_async(float* smem, const float* g) {
        if (!RD_DBG_SHARED(smem, 16, kSiteCopyDst)) return;
        const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(g) : "memory");
    }
    // copy only where ``pred`` holds (no branch)
    __device__ __forceinline__ static void cp_async_if(float* smem, const float* g, int pred) {
        if (pred && !RD_DBG_SHARED(smem, 16, kSiteCopyDst)) return;
        const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n"
                     " @p cp.async.cg.shared.global [%0], [%1], 16;\n}\n" ::"r"(s), "l"(g),
                     "r"(pred)
                     : "memory");
    }
    // one element (4 bytes), asynchronously
    __device__ __forceinline__ static void cp_async_elem(float* smem, const float* g) {
        if (!RD_DBG_SHARED(smem, 4, kSiteCopyDst)) return;
        const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(g) : "memory");
    }
};

template <> struct Store<__nv_bfloat16> {
    __device__ __forceinline__ static void load(const __nv_bfloat16* p, float (&v)[4]) {
        if (!RD_DBG_ANY(p, 8, kSiteSharedLoad)) { v[0] = v[1] = v[2] = v[3] = 0.0f; return; }
        const uint2 t = *reinterpret_cast<const uint2*>(p);
        v[0] = __uint_as_float(t.x << 16);
        v[1] = __uint_as_float(t.x & 0xffff0000u);
        v[2] = __uint_as_float(t.y << 16);
        v[3] = __uint_as_float(t.y & 0xffff0000u);
    }
    __device__ __forceinline__ static void store(__nv_bfloat16* p, const float (&v)[4]) {
        if (!RD_DBG_ANY(p, 8, kSiteSharedStore)) return;
        __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
        __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
        *reinterpret_cast<uint2*>(p) =
            make_uint2(*reinterpret_cast<unsigned*>(&a), *reinterpret_cast<unsigned*>(&b));
    }
    __device__ __forceinline__ static float get(const __nv_bfloat16* p) {
        if (!RD_DBG_ANY(p, 2, kSiteSharedLoad)) return 0.0f;
        return __bfloat162float(*p);
    }
    __device__ __forceinline__ static float round(float x) {
        return __bfloat162float(__float2bfloat16_rn(x));
    }
    __device__ __forceinline__ static void cp_async(__nv_bfloat16* smem, const __nv_bfloat16* g) {
        if (!RD_DBG_SHARED(smem, 8, kSiteCopyDst)) return;
        const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(g) : "memory");
    }
    // 2-byte elements have no asynchronous copy: element copies are plain
    __device__ __forceinline__ static void cp_async_elem(__nv_bfloat16* smem,
                                                         const __nv_bfloat16* g) {
        if (!RD_DBG_SHARED(smem, 2, kSiteCopyDst)) return;
        *smem = *g;
    }
    __device__ __forceinline__ static void cp_async_if(__nv_bfloat16* smem,
                                                       const __nv_bfloat16* g, int pred) {
        if (pred && !RD_DBG_SHARED(smem, 8, kSiteCopyDst)) return;
        const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n"
                     " @p cp.async.ca.shared.global [%0], [%1], 8;\n}\n" ::"r"(s), "l"(g),
                     "r"(pred)
                     : "memory");
    }
};

__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__host__ __device__ __forceinline__ int wrapi(int i, int n) {
    int r = i % n;
    return r < 0 ? r + n : r;
}

// Entry z of the Courant table ``tab`` (0 without a table).
__device__ __forceinline__ float courant_at(const InstDesc& sd, const float* tab, int z) {
    if (!tab || !RD_DBG_GLOBAL(sd, tab + z, 4, kSiteTable)) return 0.0f;
    return tab[z];
}

// ----------------------------------------------------------------- models
// Per-cell pieces of eq. (1).  ``react`` returns dt * R_s(c) per species.
struct MDiffusion {
    static constexpr int S = 1;
    static constexpr bool CH = false;
    template <class V>
    __device__ __forceinline__ static void react(const InstDesc&, const V*, V* inc) {
        inc[0] = vset<V>(0.0f);
    }
};

// Brusselator: R_u = a - (b+1) u + u^2 v, R_v = b u - u^2 v.
// p[0] = a, p[1] = b + 1, p[2] = b.
struct MBrusselator {
    static constexpr int S = 2;
    static constexpr bool CH = false;
    template <class V>
    __device__ __forceinline__ static void react(const InstDesc& d, const V* c, V* inc) {
        const V u = c[0], v = c[1];
        const V uuv = vmul_rounded(vmul(u, u), v);
        const V f = vadd(vfma(vset<V>(-d.p[1]), u, vset<V>(d.p[0])), uuv);
        const V g = vsub(vmul_rounded(vset<V>(d.p[2]), u), uuv);
        inc[0] = vmul(vset<V>(d.dt), f);
        inc[1] = vmul(vset<V>(d.dt), g);
    }
};

// Photochemistry NO, NO2, O3: NO2 -> NO + O3 (j), NO + O3 -> NO2 (k).
// p[0] = j, p[1] = k.
struct MAir {
    static constexpr int S = 3;
    static constexpr bool CH = false;
    template <class V>
    __device__ __forceinline__ static void react(const InstDesc& d, const V* c, V* inc) {
        const V ph = vmul_rounded(vset<V>(d.p[0]), c[1]);
        const V ti = vmul_rounded(vmul(vset<V>(d.p[1]), c[0]), c[2]);
        const V net = vmul(vset<V>(d.dt), vsub(ph, ti));
        inc[0] = net;
        inc[1] = vneg(net);
        inc[2] = net;
    }
};

// Models with a Cahn-Hilliard species (species 2, c) share one shape: the
// chemical potential mu = g(c) - p[2] Lap_h c, where Lap_h c = (sum of the
// 6 neighbours - 6 c) is the Laplacian times h^2, and the update
// c += p[1] Lap_h mu + dt R_c, with no Fickian term for c (the biharmonic
// as "Laplacian, boundary rule, Laplacian", Section 4.1).

// Front a + b -> c with Cahn-Hilliard c.
// p[0] = dt k, p[1] = dt M / h^2, p[2] = kappa / h^2.
struct MChFront {
    static constexpr int S = 3;
    static constexpr bool CH = true;
    template <class V>
    __device__ __forceinline__ static void react(const InstDesc& d, const V* c, V* inc) {
        const V q = vmul(vmul(vset<V>(d.p[0]), c[0]), c[1]);
        inc[0] = vneg(q);
        inc[1] = vneg(q);
        inc[2] = q;
    }
    // g(c) = f'(c) = 2c(c-1)(2c-1), the derivative of the double well
    template <class V> __device__ __forceinline__ static V g(const InstDesc&, V c) {
        const V c2 = vadd(c, c);
        return vmul(vmul(c2, vadd(c, vset<V>(-1.0f))), vadd(c2, vset<V>(-1.0f)));
    }
};

// The phase separation behind a front of Table 1 (row 3): c1 + c2 -> c3 at
// k1 c1 c2, the sink k2 c1 c3 taken from c1 and c3, and
// dc3/dt += -lambda Lap(eps c3 - gamma c3^3 + sigma Lap c3).
// p[0] = dt k1, p[1] = -dt lambda / h^2, p[2] = -sigma / h^2, p[3] = dt k2,
// p[4] = eps, p[5] = gamma.
struct MChTable1 {
    static constexpr int S = 3;
    static constexpr bool CH = true;
    template <class V>
    __device__ __forceinline__ static void react(const InstDesc& d, const V* c, V* inc) {
        const V q1 = vmul_rounded(vmul(vset<V>(d.p[0]), c[0]), c[1]);
        const V q2 = vmul_rounded(vmul(vset<V>(d.p[3]), c[0]), c[2]);
        inc[0] = vneg(vadd(q1, q2));
        inc[1] = vneg(q1);
        inc[2] = vsub(q1, q2);
    }
    // g(c) = eps c - gamma c^3
    template <class V> __device__ __forceinline__ static V g(const InstDesc& d, V c) {
        return vmul(c, vfma(vset<V>(-d.p[5]), vmul(c, c), vset<V>(d.p[4])));
    }
};

// dt R_s(c) of the thread's 4 cells
template <class M, int S>
__device__ __forceinline__ void react4(const InstDesc& d, const float (&c)[S][kVEC],
                                       float (&inc)[S][kVEC]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float2 cv[S], iv[S];
#pragma unroll
        for (int s = 0; s < S; ++s) cv[s] = pair_of(c[s], h);
        M::react(d, cv, iv);
#pragma unroll
        for (int s = 0; s < S; ++s) set_pair(inc[s], h, iv[s]);
    }
}

// One cell (or pair) of eq. (5) for a species with Fickian transport:
// c + inc + sum_a k_a (c[-1] + c[+1] - 2c), k_a = D_a dt / h^2; sx, sy, sz
// are the sums of the two neighbours along each axis.
template <class V>
__device__ __forceinline__ V euler_cell(V c, V sx, V sy, V sz, float kx, float ky, float kz,
                                        V inc) {
    const V c2 = vadd(c, c);
    inc = vfma(vset<V>(kz), vsub(sz, c2), inc);
    inc = vfma(vset<V>(ky), vsub(sy, c2), inc);
    inc = vfma(vset<V>(kx), vsub(sx, c2), inc);
    return vadd(c, inc);
}

// Sum of the 6 neighbours - 6 c
template <class V> __device__ __forceinline__ V lap7_cell(V c, V sx, V sy, V sz) {
    return vfma(vset<V>(-6.0f), c, vadd(vadd(sx, sy), sz));
}

// euler_cell for equal diffusivities on the three axes (k = D dt / h^2):
// c + inc + k (sum of the 6 neighbours - 6 c).
template <class V>
__device__ __forceinline__ V euler_cell_iso(V c, V sx, V sy, V sz, float k, V inc) {
    return vadd(c, vfma(vset<V>(k), lap7_cell(c, sx, sy, sz), inc));
}

// The neighbour sums of the thread's cells 2h, 2h + 1.  The x neighbours of
// a pair are no aligned pair of registers, so that sum is taken cell by cell.
__device__ __forceinline__ float2 xsum_of(const float (&xm)[kVEC], const float (&xp)[kVEC],
                                          int h) {
    return make_float2(__fadd_rn(xm[2 * h], xp[2 * h]), __fadd_rn(xm[2 * h + 1], xp[2 * h + 1]));
}

// 4 cells of euler_cell_iso
__device__ __forceinline__ void euler4_iso(const float (&c)[kVEC], const float (&xm)[kVEC],
                                           const float (&xp)[kVEC], const float (&ym)[kVEC],
                                           const float (&yp)[kVEC], const float (&zm)[kVEC],
                                           const float (&zp)[kVEC], float k,
                                           const float (&inc)[kVEC], float (&o)[kVEC]) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
        set_pair(o, h, euler_cell_iso(pair_of(c, h), xsum_of(xm, xp, h),
                                      vadd(pair_of(ym, h), pair_of(yp, h)),
                                      vadd(pair_of(zm, h), pair_of(zp, h)), k, pair_of(inc, h)));
}

// 4 cells of euler_cell
__device__ __forceinline__ void euler4_aniso(const float (&c)[kVEC], const float (&xm)[kVEC],
                                             const float (&xp)[kVEC], const float (&ym)[kVEC],
                                             const float (&yp)[kVEC], const float (&zm)[kVEC],
                                             const float (&zp)[kVEC], float kx, float ky, float kz,
                                             const float (&inc)[kVEC], float (&o)[kVEC]) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
        set_pair(o, h, euler_cell(pair_of(c, h), xsum_of(xm, xp, h),
                                  vadd(pair_of(ym, h), pair_of(yp, h)),
                                  vadd(pair_of(zm, h), pair_of(zp, h)), kx, ky, kz,
                                  pair_of(inc, h)));
}

// 4 cells of a species with any diffusivities: euler_cell_iso where they are
// equal, else euler_cell
__device__ __forceinline__ void euler4(const float (&c)[kVEC], const float (&xm)[kVEC],
                                       const float (&xp)[kVEC], const float (&ym)[kVEC],
                                       const float (&yp)[kVEC], const float (&zm)[kVEC],
                                       const float (&zp)[kVEC], float kx, float ky, float kz,
                                       const float (&inc)[kVEC], float (&o)[kVEC]) {
    if (kx == ky && kx == kz) euler4_iso(c, xm, xp, ym, yp, zm, zp, kx, inc, o);
    else euler4_aniso(c, xm, xp, ym, yp, zm, zp, kx, ky, kz, inc, o);
}

// mu = g(c) - p[2] (sum of 6 neighbours - 6 c) of the thread's 4 cells
template <class M>
__device__ __forceinline__ void mu4(const InstDesc& d, const float (&c)[kVEC],
                                    const float (&xm)[kVEC], const float (&xp)[kVEC],
                                    const float (&ym)[kVEC], const float (&yp)[kVEC],
                                    const float (&zm)[kVEC], const float (&zp)[kVEC],
                                    float (&mu)[kVEC]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 cc = pair_of(c, h);
        const float2 lap = lap7_cell(cc, xsum_of(xm, xp, h),
                                     vadd(pair_of(ym, h), pair_of(yp, h)),
                                     vadd(pair_of(zm, h), pair_of(zp, h)));
        set_pair(mu, h, vfma(vset<float2>(-d.p[2]), lap, M::g(d, cc)));
    }
}

// c + inc + pm (sum of the 6 neighbours of mu - 6 mu): the Cahn-Hilliard
// species' update on 4 cells, pm = p[1]
__device__ __forceinline__ void euler4_ch(float pm, const float (&c)[kVEC], const float (&m)[kVEC],
                                          const float (&xm)[kVEC], const float (&xp)[kVEC],
                                          const float (&ym)[kVEC], const float (&yp)[kVEC],
                                          const float (&zm)[kVEC], const float (&zp)[kVEC],
                                          const float (&inc)[kVEC], float (&o)[kVEC]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 lap = lap7_cell(pair_of(m, h), xsum_of(xm, xp, h),
                                     vadd(pair_of(ym, h), pair_of(yp, h)),
                                     vadd(pair_of(zm, h), pair_of(zp, h)));
        set_pair(o, h, vadd(pair_of(c, h), vfma(vset<float2>(pm), lap, pair_of(inc, h))));
    }
}

// ------------------------------------------------------- shared-memory map
// Every level keeps its planes in shared memory; slots are the low bits of
// the plane index.  Level 0 is a ring of 8 planes per species, P of them in
// flight ahead of the plane being consumed; an inner level has 4 plane
// buffers (a mu level holds one field).  The z neighbours a thread needs
// are its own position in planes q-1 and q+1, which it wrote (or copied)
// itself; only the x/y neighbours in plane q come from other threads, and
// that plane was completed before the last barrier.  Hence one barrier per
// plane suffices when
//   level 0:  P <= 8 - 3 (read up to two planes after arrival; the
//             Cahn-Hilliard state level reads it three planes after: P <= 4)
//   inner:    4 buffers (read up to three planes after it is written).
// Each plane is rows(ty) rows of kRW elements plus a kVEC guard at both ends.
template <class M, class ST, int T> struct Layout {
    static constexpr int S = M::S;
    static constexpr bool CH = M::CH;
    static constexpr int L = CH ? 2 * T : T;
    static constexpr int RING0 = 8;
    static constexpr int P = CH ? 4 : 5;     // level-0 planes in flight
    static constexpr int NBUF = 4;           // planes of an inner level
    __host__ __device__ static constexpr bool is_mu(int l) { return CH && (l & 1); }
    __host__ __device__ static int rows(int ty) { return ty + 2 * L; }
    __host__ __device__ static int plane_elems(int ty) { return rows(ty) * kRW + 2 * kVEC; }
    __host__ __device__ static size_t level_bytes(int l, int ty) {
        const size_t pe = plane_elems(ty);
        if (l == 0) return (size_t)RING0 * S * pe * sizeof(ST);
        if (is_mu(l)) return (size_t)NBUF * pe * sizeof(float);
        return (size_t)NBUF * S * pe * sizeof(ST);
    }
    __host__ __device__ static size_t level_offset(int l, int ty) {
        size_t o = 0;
        for (int i = 0; i < l; ++i) o += level_bytes(i, ty);
        return o;
    }
    __host__ __device__ static size_t total(int ty) { return level_offset(L, ty); }
    __host__ __device__ static int threads(int ty) { return kNQ * rows(ty); }
};

// Per-thread geometry of a work item (fixed for the whole march).
struct Pos {
    int own;          // shared-memory element offset of the thread's vector
    int offm, offp;   // vector above / below (own vector at a zero-flux y face)
    int offl;         // element left of the vector (own element 0 at x = 0)
    int xs, y;        // global x of element 0 and global y (unwrapped)
    int xhi;          // element holding x = nx-1 at a zero-flux face, else -1
};

// 7-point neighbourhood of the thread's vector in one level: centre and the
// z neighbours from planes Pc / Pm / Pp at the thread's own position, x and
// y neighbours from plane Pc.
template <class E>
__device__ __forceinline__ void gather7(const E* Pc, const E* Pm, const E* Pp, const Pos& ps,
                                        float (&c)[kVEC], float (&xm)[kVEC], float (&xp)[kVEC],
                                        float (&ym)[kVEC], float (&yp)[kVEC],
                                        float (&zm)[kVEC], float (&zp)[kVEC]) {
    Store<E>::load(Pc + ps.own, c);
    Store<E>::load(Pm + ps.own, zm);
    Store<E>::load(Pp + ps.own, zp);
    Store<E>::load(Pc + ps.offm, ym);
    Store<E>::load(Pc + ps.offp, yp);
    const float left = Store<E>::get(Pc + ps.offl);
    const float right = Store<E>::get(Pc + ps.own + kVEC);
#pragma unroll
    for (int e = 0; e < kVEC; ++e) {
        xm[e] = e ? c[e - 1] : left;
        xp[e] = (e < kVEC - 1) ? c[e + 1] : right;
    }
    if (ps.xhi >= 0) {
#pragma unroll
        for (int e = 0; e < kVEC; ++e)
            if (e == ps.xhi) xp[e] = c[e];
    }
}

// The instance a work item belongs to: the launch's own descriptor (kernel
// parameter space, read as constants) for single-instance launches, else a
// shared-memory copy of the batch entry.
template <bool ONE>
__device__ __forceinline__ const InstDesc& desc_of(const LaunchArgs& a, const InstDesc& copy) {
    if constexpr (ONE) return a.one;
    else return copy;
}

// Fetch the descriptor of the instance owning ``item`` into ``copy`` (batch
// launches); one barrier-separated pass per change of instance.  Every item
// below nitems has exactly one owner, whose thread alone writes s_inst: it
// needs no initial value, and a store of one by another warp could land after
// the owner's.
__device__ __forceinline__ void load_desc(const LaunchArgs& a, long long item, InstDesc& copy,
                                          int& s_inst, int& cur_inst) {
    const int tid = threadIdx.x;
    for (int i = tid; i < a.ninst; i += blockDim.x) {
        const long long b0 = a.desc[i].item_begin;
        const long long b1 = (i + 1 < a.ninst) ? a.desc[i + 1].item_begin : a.nitems;
        if (item >= b0 && item < b1) s_inst = i;
    }
    __syncthreads();
    if (s_inst != cur_inst) {
        cur_inst = s_inst;
        const int* src = reinterpret_cast<const int*>(a.desc + cur_inst);
        int* dst = reinterpret_cast<int*>(&copy);
        for (int i = tid; i < (int)(sizeof(InstDesc) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
}

// Work items of a CTA.  A single instance's items cost the same, so a CTA
// takes every gridDim-th one; a batch's may differ (partial tiles, short
// last z-chunks, unequal instances), so when the host passes the batch's
// counter (a.work) its CTAs pull the next item as they finish one.  Each CTA's last pull fails (its
// ticket is at least nitems); the CTA holding the launch's last ticket,
// nitems + gridDim - 1, pulls after every other CTA has finished its
// items, so it also counts the launch as completed (work[1]) and zeroes
// the item counter for the next launch.  Called by every thread of the CTA
// together; the item loops end with a block barrier, so s_item is free to
// overwrite.
__device__ __forceinline__ long long pull_item(const LaunchArgs& a, long long& s_item) {
    if (threadIdx.x == 0) {
        const unsigned long long t = atomicAdd(a.work, 1ull);
        if (t == (unsigned long long)a.nitems + gridDim.x - 1) {
            atomicAdd(a.work + 1, 1ull);
            atomicExch(a.work, 0ull);
        }
        s_item = (long long)t;
    }
    __syncthreads();
    return s_item;
}
// A batch member whose launches for the current step call are used up
// (rd_batch_step_each) is left alone: its items are skipped, its fields
// keep the level its last step wrote.  The same for every thread.
template <bool ONE>
__device__ __forceinline__ bool member_done(const LaunchArgs& a, const InstDesc& sd) {
    if (ONE || !a.work || sd.launch_cap < 0) return false;
    return (long long)a.work[1] >= sd.launch_cap;
}
template <bool ONE>
__device__ __forceinline__ long long first_item(const LaunchArgs& a, long long& s_item) {
    if (ONE || !a.work) return blockIdx.x;
    return pull_item(a, s_item);
}
template <bool ONE>
__device__ __forceinline__ long long next_item(const LaunchArgs& a, long long item,
                                               long long& s_item) {
    if (ONE || !a.work) return item + gridDim.x;
    return pull_item(a, s_item);
}

// Held (Dirichlet) layers: the first face in -x,+x,-y,+y,-z,+z wins.
__device__ __forceinline__ void held_layers(const InstDesc& sd, int s, int xs, int y, int q,
                                            float (&o)[kVEC]) {
    const unsigned hm = sd.held_mask[s];
    if (!hm) return;
#pragma unroll
    for (int e = 0; e < kVEC; ++e) {
        const int x = xs + e;
        float hv = o[e];
        if ((hm & 32u) && q == sd.nz - 1) hv = sd.held_val[s][5];
        if ((hm & 16u) && q == 0) hv = sd.held_val[s][4];
        if ((hm & 8u) && y == sd.ny - 1) hv = sd.held_val[s][3];
        if ((hm & 4u) && y == 0) hv = sd.held_val[s][2];
        if ((hm & 2u) && x == sd.nx - 1) hv = sd.held_val[s][1];
        if ((hm & 1u) && x == 0) hv = sd.held_val[s][0];
        o[e] = hv;
    }
}

// Faces of the grid that a thread's 4 cells (x = xs..xs+3, row y, plane
// q) lie on, as bits in the order of held_mask: -x, +x, -y, +y, -z, +z.
__device__ __forceinline__ unsigned xy_faces(int xs, int y, int nx, int ny) {
    return (xs <= 0 && xs + kVEC > 0 ? 1u : 0u) | (xs <= nx - 1 && xs + kVEC > nx - 1 ? 2u : 0u) |
           (y == 0 ? 4u : 0u) | (y == ny - 1 ? 8u : 0u);
}
__device__ __forceinline__ unsigned z_faces(int q, int nz) {
    return (q == 0 ? 16u : 0u) | (q == nz - 1 ? 32u : 0u);
}

// held_layers for a thread whose face bits are known: the same result, the
// per-cell tests run only where a held face is touched
__device__ __forceinline__ void held_layers_at(const InstDesc& sd, int s, unsigned faces, int xs,
                                               int y, int q, float (&o)[kVEC]) {
    if (sd.held_mask[s] & faces) {
        asm volatile("");   // keep the branch: few vectors touch a held face
        held_layers(sd, s, xs, y, q, o);
    }
}

// First-order upwind along one axis with Courant number cu = u dt / h:
// in -= cu (c - c[-1]) for cu > 0, cu (c[+1] - c) for cu < 0 (Section 4.1).
__device__ __forceinline__ void upwind_axis(float cu, const float (&c)[kVEC],
                                            const float (&cm)[kVEC], const float (&cp)[kVEC],
                                            float (&in)[kVEC]) {
    if (cu > 0.0f) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            set_pair(in, h, vfma(vset<float2>(-cu), vsub(pair_of(c, h), pair_of(cm, h)),
                                 pair_of(in, h)));
    } else if (cu < 0.0f) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            set_pair(in, h, vfma(vset<float2>(-cu), vsub(pair_of(cp, h), pair_of(c, h)),
                                 pair_of(in, h)));
    }
}

// Courant numbers along y and z of the 3-D wind for the launch reading time
// level ``lin`` (zero without it): u_z = wz_amp sin(n wz_omega) at the step
// index n of that level, evaluated in double precision.  The CTA taking an
// instance's first work item also records n + 1 as the step index of the
// level it writes (read by the next launch, never by this one).
__device__ __forceinline__ void wind3d(const InstDesc& sd, int lin, long long local, float& cy,
                                       float& cz) {
    cy = 0.0f;
    cz = 0.0f;
    if (!sd.stepn) return;
    if (!RD_DBG_GLOBAL(sd, sd.stepn, 16, kSiteTable)) return;
    const long long n = sd.stepn[lin];
    cy = sd.cy;
    cz = (float)(sd.wz_amp * sin((double)n * sd.wz_omega));
    if (local == 0 && threadIdx.x == 0) sd.stepn[lin ^ 1] = n + 1;
}

// New value of one species on the thread's 4 cells (eq. (5)): reaction
// increment ``inc`` (dt R), point source, upwind advection, Fickian
// transport; held layers are applied by the caller.  Shared by every
// kernel so that all launch shapes give identical bits.
__device__ __forceinline__ void species_core(const InstDesc& sd, int s, const float (&c)[kVEC],
                                             const float (&xm)[kVEC], const float (&xp)[kVEC],
                                             const float (&ym)[kVEC], const float (&yp)[kVEC],
                                             const float (&zm)[kVEC], const float (&zp)[kVEC],
                                             const float (&inc)[kVEC], float cx, bool src_here,
                                             bool px, int xs, float (&o)[kVEC], float cy = 0.0f,
                                             float cz = 0.0f) {
    const float kx = sd.kx[s], ky = sd.ky[s], kz = sd.kz[s];
    const bool src_s = src_here && s == sd.src_s;
    // every test below is uniform over the 4 cells: taken once, not per cell
    float in[kVEC];
#pragma unroll
    for (int e = 0; e < kVEC; ++e) in[e] = inc[e];
    if (src_s) {
#pragma unroll
        for (int e = 0; e < kVEC; ++e)
            if ((px ? wrapi(xs + e, sd.nx) : xs + e) == sd.src_x) in[e] = __fadd_rn(in[e], sd.src_amt);
    }
    // first-order upwind advection, Courant number cx = u dt / h; the x
    // differences cell by cell (see xsum_of)
    if (cx > 0.0f) {
#pragma unroll
        for (int e = 0; e < kVEC; ++e) in[e] = __fmaf_rn(-cx, __fsub_rn(c[e], xm[e]), in[e]);
    } else if (cx < 0.0f) {
#pragma unroll
        for (int e = 0; e < kVEC; ++e) in[e] = __fmaf_rn(-cx, __fsub_rn(xp[e], c[e]), in[e]);
    }
    // the same along y and z (the 3-D wind of Table 1, row 4)
    upwind_axis(cy, c, ym, yp, in);
    upwind_axis(cz, c, zm, zp, in);
    euler4(c, xm, xp, ym, yp, zm, zp, kx, ky, kz, in, o);
}

// species_core followed by the held layers
__device__ __forceinline__ void species_update(const InstDesc& sd, int s, const float (&c)[kVEC],
                                               const float (&xm)[kVEC], const float (&xp)[kVEC],
                                               const float (&ym)[kVEC], const float (&yp)[kVEC],
                                               const float (&zm)[kVEC], const float (&zp)[kVEC],
                                               const float (&inc)[kVEC], float cx, bool src_here,
                                               bool px, int xs, int y, int q, float (&o)[kVEC]) {
    species_core(sd, s, c, xm, xp, ym, yp, zm, zp, inc, cx, src_here, px, xs, o);
    held_layers(sd, s, xs, y, q, o);
}

// ------------------------------------------------------------------ kernel
template <class M, class ST, int T, bool ONE>
__global__ void __launch_bounds__(kMaxThreads, 2) rd_step_kernel(const __grid_constant__ LaunchArgs a) {
    using LY = Layout<M, ST, T>;
    constexpr int S = M::S;
    constexpr bool CH = M::CH;
    constexpr int L = LY::L;
    constexpr int P = LY::P;

    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ InstDesc sdm;
    __shared__ int s_inst;
    __shared__ long long s_item;

    const int tid = threadIdx.x;
    const int TY = a.ty;
    const int NR = LY::rows(TY);
    const int PE = LY::plane_elems(TY);
    const int r = tid / kNQ;             // row of the thread's position
    const int v = tid - r * kNQ;         // vector of the thread's position

    // plane X of state level m, species s; plane X of mu level m
    auto state_plane = [&](int m, int s, int X) -> ST* {
        const int slot = (m == 0) ? (X & (LY::RING0 - 1)) : (X & (LY::NBUF - 1));
        return reinterpret_cast<ST*>(smem + LY::level_offset(m, TY)) + (size_t)(slot * S + s) * PE +
               kVEC;
    };
    auto mu_plane = [&](int m, int X) -> float* {
        return reinterpret_cast<float*>(smem + LY::level_offset(m, TY)) +
               (size_t)(X & (LY::NBUF - 1)) * PE + kVEC;
    };

    int cur_inst = -1;
    for (long long item = first_item<ONE>(a, s_item); item < a.nitems;
         item = next_item<ONE>(a, item, s_item)) {
        if constexpr (!ONE) load_desc(a, item, sdm, s_inst, cur_inst);
        const InstDesc& sd = desc_of<ONE>(a, sdm);
        if (member_done<ONE>(a, sd)) continue;   // block-uniform

        const int nx = sd.nx, ny = sd.ny, nz = sd.nz;
        const bool px = sd.per_x, py = sd.per_y, pz = sd.per_z;
        const long long local = item - sd.item_begin;
        const int txi = (int)(local % sd.ntx);
        const int tyi = (int)((local / sd.ntx) % sd.nty);
        const int zc = (int)(local / ((long long)sd.ntx * sd.nty));
        const int x0 = txi * kTileQ * kVEC, y0 = tyi * TY;
        const int z0 = zc * sd.zchunk;
        const int z1 = min(z0 + sd.zchunk, nz);
        const int lin = sd.par ^ a.parity;

        // ---- per-thread geometry
        Pos ps;
        ps.y = y0 - L + r;
        ps.xs = x0 - kVEC + v * kVEC;
        const bool yin = py || (ps.y >= 0 && ps.y < ny);
        const bool xin = px || (ps.xs + kVEC > 0 && ps.xs < nx);
        const bool in_dom = r < NR && yin && xin;
        ps.own = r * kRW + v * kVEC;
        ps.offm = (!py && ps.y == 0) ? ps.own : ps.own - kRW;
        ps.offp = (!py && ps.y == ny - 1) ? ps.own : ps.own + kRW;
        ps.offl = (!px && ps.xs == 0) ? ps.own : ps.own - 1;
        ps.xhi = (!px && ps.xs <= nx - 1 && nx - 1 < ps.xs + kVEC) ? nx - 1 - ps.xs : -1;
        const int yw = py ? wrapi(ps.y, ny) : ps.y;
        // global load of the thread's vector: 1 = one copy, 2 = wrapped
        // element by element, 0 = none
        int ld_mode = 0;
        long long ld_off = 0;
        if (in_dom) {
            const long long row = (long long)yw * sd.pitch;
            if (ps.xs >= 0 && ps.xs < nx && (!px || ps.xs + kVEC <= nx)) {
                ld_mode = 1;
                ld_off = row + ps.xs;
            } else if (px) {
                const int xw = wrapi(ps.xs, nx);
                if (xw % kVEC == 0 && xw + kVEC <= nx) { ld_mode = 1; ld_off = row + xw; }
                else { ld_mode = 2; ld_off = row; }
            }
        }
        // levels this position computes: bit l (l = L: the stored tile)
        unsigned lbits = 0;
        if (in_dom) {
#pragma unroll
            for (int l = 1; l < L; ++l)
                if (r >= l && r < NR - l) lbits |= 1u << l;
            if (r >= L && r < L + TY && v >= 1 && v <= kTileQ && ps.y >= 0 && ps.y < ny &&
                ps.xs < nx)
                lbits |= 1u << L;
        }
        const long long st_off = (long long)ps.y * sd.pitch + ps.xs;
        const bool src_col = sd.src_s >= 0 && yw == sd.src_y;

        // ---- loads: plane ``nld`` (wrapped index zld) into the level-0 ring
        const int pbeg = z0 - L, pend = z1 + L;
        int nld = pbeg;
        int zld = pz ? wrapi(nld, nz) : nld;
        auto issue = [&]() {
            if (nld < pend && ld_mode != 0 && (pz || (nld >= 0 && nld < nz))) {
                const long long zoff = (long long)zld * sd.plane + ld_off;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const ST* g = reinterpret_cast<const ST*>(sd.base[lin][s]) + zoff;
                    ST* dst = state_plane(0, s, nld) + ps.own;
                    if (ld_mode == 1) {
                        if (RD_DBG_GLOBAL(sd, g, 4 * (int)sizeof(ST), kSiteCopySrc))
                            Store<ST>::cp_async(dst, g);
                    } else {
#pragma unroll
                        for (int e = 0; e < kVEC; ++e) {
                            const ST* ge = g + wrapi(ps.xs + e, nx);
                            if (RD_DBG_GLOBAL(sd, ge, (int)sizeof(ST), kSiteCopySrc) &&
                                RD_DBG_SHARED(dst + e, (int)sizeof(ST), kSiteCopyDst))
                                dst[e] = *ge;
                        }
                    }
                }
            }
            ++nld;
            if (!pz) zld = nld;
            else if (++zld == nz) zld = 0;
            cp_async_commit();
        };

#pragma unroll 1
        for (int j = 0; j < P; ++j) issue();
        int zcur = pz ? wrapi(pbeg, nz) : pbeg;   // wrapped index of plane p
#pragma unroll 1
        for (int p = pbeg; p < pend; ++p) {
            issue();
            cp_async_wait<P>();
            __syncthreads();
#pragma unroll
            for (int l = 1; l <= L; ++l) {
                const int q = p - l;
                const bool valid = q >= z0 - L + l && q < z1 + L - l && (pz || (q >= 0 && q < nz));
                if (!valid || !(lbits & (1u << l))) continue;
                const bool fin = (l == L);
                int zw = q;
                if (pz) { zw = zcur - l; while (zw < 0) zw += nz; }
                // z neighbours: the face plane itself at a zero-flux z face
                const int qm = (!pz && q == 0) ? q : q - 1;
                const int qp = (!pz && q == nz - 1) ? q : q + 1;
                if constexpr (CH) {
                    if (LY::is_mu(l)) {
                        // mu of the Cahn-Hilliard species from state level l-1
                        float c[kVEC], xm[kVEC], xp[kVEC], ym[kVEC], yp[kVEC], zm[kVEC], zp[kVEC];
                        gather7<ST>(state_plane(l - 1, 2, q), state_plane(l - 1, 2, qm),
                                    state_plane(l - 1, 2, qp), ps, c, xm, xp, ym, yp, zm, zp);
                        float mo[kVEC];
                        mu4<M>(sd, c, xm, xp, ym, yp, zm, zp, mo);
                        Store<float>::store(mu_plane(l, q) + ps.own, mo);
                        continue;
                    }
                }
                // state update from level ls (and, for Cahn-Hilliard, mu at l-1)
                const int ls = CH ? l - 2 : l - 1;
                float inc[S][kVEC];
                {
                    float cen[S][kVEC];
#pragma unroll
                    for (int s = 0; s < S; ++s) Store<ST>::load(state_plane(ls, s, q) + ps.own, cen[s]);
                    react4<M>(sd, cen, inc);
                }
                const float cx = courant_at(sd, sd.courant, zw);
                const bool src_here = src_col && zw == sd.src_z;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    float o[kVEC];
                    if (CH && s == 2) {
                        // c += dt M / h^2 * (7-point Laplacian of mu)
                        float m0[kVEC], mxm[kVEC], mxp[kVEC], mym[kVEC], myp[kVEC], mzm[kVEC],
                            mzp[kVEC], c[kVEC];
                        gather7<float>(mu_plane(l - 1, q), mu_plane(l - 1, qm), mu_plane(l - 1, qp),
                                       ps, m0, mxm, mxp, mym, myp, mzm, mzp);
                        Store<ST>::load(state_plane(ls, 2, q) + ps.own, c);
                        euler4_ch(sd.p[1], c, m0, mxm, mxp, mym, myp, mzm, mzp, inc[s], o);
                    } else {
                        float c[kVEC], xm[kVEC], xp[kVEC], ym[kVEC], yp[kVEC], zm[kVEC], zp[kVEC];
                        gather7<ST>(state_plane(ls, s, q), state_plane(ls, s, qm),
                                    state_plane(ls, s, qp), ps, c, xm, xp, ym, yp, zm, zp);
                        species_update(sd, s, c, xm, xp, ym, yp, zm, zp, inc[s], cx, src_here, px,
                                       ps.xs, ps.y, q, o);
                    }
                    if (CH && s == 2) held_layers(sd, s, ps.xs, ps.y, q, o);
                    if (fin) {
                        ST* g = reinterpret_cast<ST*>(sd.base[lin ^ 1][s]) +
                                (long long)q * sd.plane + st_off;
                        if (RD_DBG_GLOBAL(sd, g, 4 * (int)sizeof(ST), kSiteStateStore))
                            Store<ST>::store(g, o);
                    } else {
                        // inner level, rounded exactly as a stored state
                        Store<ST>::store(state_plane(l, s, q) + ps.own, o);
                    }
                }
            }
            if (pz && ++zcur == nz) zcur = 0;
        }
        cp_async_wait<0>();
        __syncthreads();
    }
}

// How one vector is fetched: 1 = one async copy, 2 = element by element (a
// vector that wraps round a periodic x axis; in the 8-cell kernel also one
// straddling a zero-flux face), 0 = nothing.
struct Fetch {
    int mode;
    unsigned goff;   // offset of row + x (mode 2: of the row) within a plane, in
                     // 4-cell vectors (plane_fits, rd_internal.h)
    int soff;    // byte offset of the position within a plane buffer
    int xs;      // global x of the vector's first element (unwrapped)
};

// the 4-cell vector ``v`` vectors past p
template <class ST> __host__ __device__ __forceinline__ const ST* vec_at(const ST* p, unsigned v) {
    return p + (unsigned long long)v * kVEC;
}

template <class ST>
__device__ __forceinline__ void lds_vec(const unsigned char* p, float (&v)[kVEC]) {
    Store<ST>::load(reinterpret_cast<const ST*>(p), v);
}
template <class ST>
__device__ __forceinline__ float lds_one(const unsigned char* p) {
    return Store<ST>::get(reinterpret_cast<const ST*>(p));
}

}  // namespace rdk

#include "rd_step1w_kernel.cuh"
#include "rd_march_kernel.cuh"
#include "rd_stepch_kernel.cuh"

namespace rdk {

// Whether T steps per launch at tile height ty run the two-step kernel
// (whole inner warps: even heights; its CTA size); else the multi-level one.
template <class M, class ST> constexpr bool two_step(int T, int ty) {
    return T == 2 && !M::CH && !(ty & 1) && LayoutM<M, ST, 2>::threads(ty) <= kMaxThreads;
}

// Launch helper used by the per-model translation units.
template <class M, class ST, int T, bool ONE>
cudaError_t launch_one(const LaunchArgs& a, int grid, size_t smem, cudaStream_t st, int* occ) {
    void (*k)(const LaunchArgs) = nullptr;
    int threads = 0;
    // which kernel, and its slot in ``configured`` below
    int variant = 0;
    bool chained = true;       // the kernels that wait for the launch before them
    if constexpr (T == 1 && M::CH) {
        k = a.plain ? rd_marchch_kernel<M, ST, ONE, true> : rd_marchch_kernel<M, ST, ONE, false>;
        threads = LayoutCH<ST>::threads(a.ty);
        variant = a.plain ? 1 : 0;
    } else if constexpr (T == 1) {
        // the march kernel needs an even tile height (16 ty inner threads as
        // whole warps); an odd one -- the last launch of a
        // call whose tuning steps 2 or 3 per launch -- runs the multi-level
        // kernel at T = 1
        const bool lean = !(a.ty & 1);
        if (lean && a.vw == 8) {   // 8 cells per thread (rd_step1w_kernel.cuh)
            k = a.plain   ? rd_step1w_kernel<M, ST, ONE, true, false>
                : a.wind3 ? rd_step1w_kernel<M, ST, ONE, false, true>
                          : rd_step1w_kernel<M, ST, ONE, false, false>;
            threads = Layout1w<M, ST>::threads(a.ty);
            variant = a.plain ? 1 : a.wind3 ? 2 : 3;
        } else if (lean) {
            k = a.plain   ? rd_march_kernel<M, ST, 1, ONE, kPlain>
                : a.wind3 ? rd_march_kernel<M, ST, 1, ONE, kWind3>
                          : rd_march_kernel<M, ST, 1, ONE, kGeneral>;
            // batches, whose members differ, keep the general variant
            const bool windx = ONE && a.windx && !a.plain && !a.wind3;
            if constexpr (ONE)
                if (windx) k = rd_march_kernel<M, ST, 1, true, kWindX>;
            threads = LayoutM<M, ST, 1>::threads(a.ty);
            variant = a.plain ? 4 : a.wind3 ? 5 : windx ? 7 : 6;
        } else {
            k = rd_step_kernel<M, ST, T, ONE>;
            threads = Layout<M, ST, T>::threads(a.ty);
            chained = false;
        }
    } else {
        k = rd_step_kernel<M, ST, T, ONE>;
        threads = Layout<M, ST, T>::threads(a.ty);
        chained = false;
        if constexpr (T == 2 && !M::CH)
            if (two_step<M, ST>(T, a.ty)) {
                chained = true;
                k = a.plain ? rd_march_kernel<M, ST, 2, ONE, kPlain>
                            : rd_march_kernel<M, ST, 2, ONE, kGeneral>;
                threads = LayoutM<M, ST, 2>::threads(a.ty);
                variant = a.plain ? 1 : 2;
            }
    }
    // dynamic shared memory granted so far, per kernel variant
    static size_t configured[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    size_t& conf = configured[variant];
    if (smem > conf) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        conf = smem;
    }
    if (threads > kMaxThreads) return cudaErrorInvalidConfiguration;
    if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, threads, smem);
    if (chained) return launch_chained(k, a, grid, threads, smem, st);
    k<<<grid, threads, smem, st>>>(a);
    return cudaGetLastError();
}

template <class M, bool ONE>
cudaError_t launch_var(int storage, int tsteps, const LaunchArgs& a, int grid, size_t smem,
                       cudaStream_t st, int* occ) {
    if (storage == RD_STORE_F32) {
        switch (tsteps) {
        case 1: return launch_one<M, float, 1, ONE>(a, grid, smem, st, occ);
        case 2: return launch_one<M, float, 2, ONE>(a, grid, smem, st, occ);
        case 3: if constexpr (!M::CH) return launch_one<M, float, 3, ONE>(a, grid, smem, st, occ);
                break;
        default: break;
        }
    } else {
        switch (tsteps) {
        case 1: return launch_one<M, __nv_bfloat16, 1, ONE>(a, grid, smem, st, occ);
        case 2: return launch_one<M, __nv_bfloat16, 2, ONE>(a, grid, smem, st, occ);
        case 3:
            if constexpr (!M::CH) return launch_one<M, __nv_bfloat16, 3, ONE>(a, grid, smem, st, occ);
            break;
        default: break;
        }
    }
    return cudaErrorInvalidValue;
}

template <class M>
cudaError_t launch_model(int storage, int tsteps, const LaunchArgs& a, int grid, size_t smem,
                         cudaStream_t st, int* occ) {
    return a.use_one ? launch_var<M, true>(storage, tsteps, a, grid, smem, st, occ)
                     : launch_var<M, false>(storage, tsteps, a, grid, smem, st, occ);
}

template <class M>
size_t smem_for(int storage, int tsteps, int ty, int vw = 4) {
    if (tsteps == 1 && !M::CH && vw == 8)
        return storage == RD_STORE_F32 ? Layout1w<M, float>::total(ty)
                                       : Layout1w<M, __nv_bfloat16>::total(ty);
    if (storage == RD_STORE_F32) {
        switch (tsteps) {
        case 1: return M::CH ? LayoutCH<float>::total(ty)
                             : (ty & 1) ? Layout<M, float, 1>::total(ty) : LayoutM<M, float, 1>::total(ty);
        case 2: if constexpr (!M::CH)
                    if (two_step<M, float>(2, ty)) return LayoutM<M, float, 2>::total(ty);
                return Layout<M, float, 2>::total(ty);
        case 3: return Layout<M, float, 3>::total(ty);
        }
    } else {
        switch (tsteps) {
        case 1: return M::CH ? LayoutCH<__nv_bfloat16>::total(ty)
                             : (ty & 1) ? Layout<M, __nv_bfloat16, 1>::total(ty)
                                        : LayoutM<M, __nv_bfloat16, 1>::total(ty);
        case 2: if constexpr (!M::CH)
                    if (two_step<M, __nv_bfloat16>(2, ty))
                        return LayoutM<M, __nv_bfloat16, 2>::total(ty);
                return Layout<M, __nv_bfloat16, 2>::total(ty);
        case 3: return Layout<M, __nv_bfloat16, 3>::total(ty);
        }
    }
    return 0;
}

}  // namespace rdk
