// rd_step19_kernel.cuh -- one forward-Euler step of eq. (5) with the
// 19-point Laplacian of eqs. (3)-(4) (sm_103a).
//
// Work items, copies, thread layout and boundary rules are those of
// rd_march_kernel at one step per launch: one thread per 4-cell vector of a
// 64 x TY tile plus one halo warp, planes of the current state copied into a
// shared-memory ring by 16-byte cp.async several planes ahead, rows holding
// every field side by side, one barrier per plane, register sets that change
// roles from plane to plane, x neighbours by warp shuffle.  What differs:
//
//  * Neighbourhood.  A cell reads the 3x3 block of its own plane (weights
//    -24 centre, 2 faces, 1 diagonals) and the 5-point cross of the planes
//    below and above (2 centre, 1 faces); corners weigh 0.
//  * Per-plane sums carried down the march.  When plane k arrives, a
//    thread forms at each of its 4 cells, with X = xm + xp + ym + yp,
//        Z_k = 2 c + X                 (plane k as a z-neighbour)
//        W_k = 2 X + the 4 diagonals   (plane k as the centre plane)
//    so that 6 h^2 Lap c on plane q = W_q - 24 c_q + Z_{q-1} + Z_{q+1}.
//    Z_{q-1}, Z_q, W_q and c_q stay in registers; each plane is read from
//    shared memory once, on arrival (plane q+1 at step q).
//  * Ring reuse.  At step q the slot of plane q-1 is refilled; its
//    neighbours were read at step q-2 (on arrival) and, with wind, q-1; the
//    sums of a work item's first two planes are formed before its first step.
//
// Measured against the kernel before it (scalar arithmetic, single-element
// shared loads with a 4-way bank conflict, sums of the field rows moved from
// register to register), best tilings: 192^3 Turing 248 -> 321 GLUPS, the
// 192^3 Cahn-Hilliard step 84 -> 120, the 144 x 144 x 384 plume 194 -> 268.
// It is bound by latency: 12 to 18 warps on an SM wait on one another's
// barrier and on shuffles and shared loads.
//
// An edge ghost composes the rules of the two axes it crosses, as the paper
// fills its edges after its faces (Section 4.1): rows beyond a zero-flux y
// face are copied in as the face row, and a thread at a zero-flux x face
// reads its own column in the rows above and below too.  A held layer's cell
// takes its bc value.
#pragma once

#include "rd_step19.h"
#include "rd_step_kernel.cuh"

namespace rdk {

// PASS 0: one step of a model without Cahn-Hilliard.  For the models with a
// Cahn-Hilliard species (species 2, c) a step is two launches, the paper's
// "Laplacian, boundary rule, Laplacian" (Section 4.1): PASS 1 writes the
// chemical potential mu = g(c) - p[2] h^2 Lap c of every cell to the
// instance's mu field, PASS 2 then updates a, b and c, reading mu as one more
// field of the ring (its ghost cells copied in under the same rules, which
// is the paper's "boundary rule" applied to mu) and adding p[1] h^2 Lap mu
// to c.  The ring of PASS 1 holds species 2 only.
template <class M, class ST, int PASS> struct Layout19 {
    static constexpr int S = M::S;
    static constexpr int NS = PASS == 1 ? 1 : S;    // state fields per row
    static constexpr bool MUF = PASS == 2;          // plus one float mu field
    static constexpr int RING = kRing19;
    static constexpr int P = RING;                  // planes issued ahead of q - 1
    static constexpr int SPB = kRW * (int)sizeof(ST);
    static constexpr int ROWB = row19_bytes(NS, (int)sizeof(ST), MUF);
    static_assert(ROWB % 16 == 0 && (NS * SPB) % 16 == 0, "16-byte vectors");
    static_assert(PASS == 0 || M::CH, "passes 1 and 2 are for Cahn-Hilliard models");
    // registers a thread may take (GLUPS at the best tilings when the budgets
    // were chosen; the kernel has gained up to 8 % since): the
    // one-species plume 250 (80) 239 (96) 231 (128); two-species Turing 192^3
    // 275 (80) 311 (96) 319 (128); the Cahn-Hilliard step 72 (80) 102 (128)
    static constexpr int regs() {
        return NS == 1 && PASS == 0 && sizeof(ST) == 4 ? 80 : 128;
    }
    __host__ __device__ static int plane_bytes(int ty) {
        return plane19_bytes(NS, (int)sizeof(ST), MUF, ty);
    }
    __host__ __device__ static size_t total(int ty) {
        return smem19_pass_bytes(NS, (int)sizeof(ST), MUF, ty);
    }
    __host__ __device__ static int threads(int ty) { return kTileQ * ty + 32; }
};

// A fetch of the own vector in one word: its offset, or kNone (positions
// outside the grid, in tiles that it does not fill, copy nothing) or kElems
// (element by element).
constexpr unsigned kNone = 0xffffffffu, kElems = 0xfffffffeu;
__host__ __device__ __forceinline__ unsigned own_offset(const Fetch& f) {
    return f.mode == 1 ? f.goff : f.mode == 2 ? kElems : kNone;
}

// Own vector c and the sums Z, W of one field's plane at the thread's 4
// cells; ``p`` points at the own vector in the ring, rows ROWB bytes apart.
// The x neighbours of a pair are no aligned pair of registers: sums along x
// are taken cell by cell, everything else packed.
template <class ST, int ROWB>
__device__ __forceinline__ void plane_sums19(const XSides& sides, const unsigned char* p,
                                             float (&c)[kVEC], float (&zs)[kVEC],
                                             float (&ws)[kVEC]) {
    float ym[kVEC], yp[kVEC], l[3], r[3];
    lds_vec<ST>(p, c);
    lds_vec<ST>(p - ROWB, ym);
    lds_vec<ST>(p + ROWB, yp);
    sides.set_ghost1(c);
    sides.set_ghost1(ym);
    sides.set_ghost1(yp);
    sides.get3<ST, ROWB>(c, ym, yp, p, l, r);
    // xm + xp of the pair h of a row with the elements le, re beside it
    auto xpair = [](const float(&v)[kVEC], float le, float re, int h) {
        return h ? make_float2(__fadd_rn(v[1], v[3]), __fadd_rn(v[2], re))
                 : make_float2(__fadd_rn(le, v[1]), __fadd_rn(v[0], v[2]));
    };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 cross =
            vadd(xpair(c, l[0], r[0], h), vadd(pair_of(ym, h), pair_of(yp, h)));
        const float2 diag = vadd(xpair(ym, l[1], r[1], h), xpair(yp, l[2], r[2], h));
        set_pair(zs, h, vfma(vset<float2>(2.0f), pair_of(c, h), cross));
        set_pair(ws, h, vfma(vset<float2>(2.0f), cross, diag));
    }
}

// New value of one species on the thread's 4 cells: c + inc + k6 * lap6,
// k6 = D dt / (6 h^2), lap6 = 6 h^2 Lap c, plus the point source and
// first-order upwind advection (Courant number cx, x neighbours from the
// own vector and the elements ``left`` / ``right`` beside it).
template <bool PLAIN>
__device__ __forceinline__ void species19(const InstDesc& sd, int s, float k6,
                                          const float (&c)[kVEC], const float (&lap6)[kVEC],
                                          const float (&inc)[kVEC], float cx, float left,
                                          float right, bool src_here, bool px, int xs,
                                          float (&o)[kVEC]) {
    float in[kVEC];
#pragma unroll
    for (int e = 0; e < kVEC; ++e) in[e] = inc[e];
    if constexpr (!PLAIN) {
        if (src_here && s == sd.src_s) {
#pragma unroll
            for (int e = 0; e < kVEC; ++e)
                if ((px ? wrapi(xs + e, sd.nx) : xs + e) == sd.src_x)
                    in[e] = __fadd_rn(in[e], sd.src_amt);
        }
        if (cx > 0.0f) {
#pragma unroll
            for (int e = 0; e < kVEC; ++e) {
                const float xm = e ? c[e - 1] : left;
                in[e] = __fmaf_rn(-cx, __fsub_rn(c[e], xm), in[e]);
            }
        } else if (cx < 0.0f) {
#pragma unroll
            for (int e = 0; e < kVEC; ++e) {
                const float xp = e < kVEC - 1 ? c[e + 1] : right;
                in[e] = __fmaf_rn(-cx, __fsub_rn(xp, c[e]), in[e]);
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
        set_pair(o, h, vadd(pair_of(c, h),
                            vfma(vset<float2>(k6), pair_of(lap6, h), pair_of(in, h))));
}

// PLAIN: no held layer, point source or wind.  PASS: see Layout19.  W3:
// the 3-D wind (upwind along y and z too; never with PLAIN, PASS 0 only).
template <class M, class ST, bool ONE, bool PLAIN, int PASS, bool W3 = false>
__global__ void __maxnreg__((Layout19<M, ST, PASS>::regs()))
rd_march19_kernel(const __grid_constant__ LaunchArgs a) {
    using LY = Layout19<M, ST, PASS>;
    constexpr int S = M::S;
    constexpr int NS = LY::NS;
    constexpr bool MUF = LY::MUF;
    // fields whose plane sums are formed: every state field (PASS 0), c
    // (PASS 1), a, b and mu (PASS 2; c needs only its own cells there)
    constexpr int NSUM = PASS == 2 ? 3 : NS;
    constexpr int P = LY::P;
    constexpr int RING = LY::RING;
    constexpr int EB = (int)sizeof(ST);
    constexpr int SPB = LY::SPB;
    constexpr int ROWB = LY::ROWB;
    constexpr unsigned FULL = 0xffffffffu;

    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ InstDesc sdm;
    __shared__ int s_inst;
    __shared__ long long s_item;

    const int tid = threadIdx.x;
    const int TY = a.ty;
    const int SLOTB = LY::plane_bytes(TY);
    const int ninner = kTileQ * TY;
    const TilePos t(min(tid, ninner + TilePos::ring(TY) - 1), TY);
    const int hl = tid - ninner;                             // >= 0: halo thread
    const bool inner = hl < 0;
    const bool inner_warp = __all_sync(FULL, inner);         // TY is even
    // byte offsets of the own vector, in the state fields and in mu, slot 0
    const int own0 = kGuard19 + t.r * ROWB + t.v * kVEC * EB;
    int4* const hfetch = reinterpret_cast<int4*>(smem + RING * SLOTB);
    const int mu_own = NS * SPB + t.v * kVEC * (4 - EB);     // from the own vector

    if constexpr (!ONE) chain_wait();   // the batch's counters are read first
    int cur_inst = -1;
    for (long long item = first_item<ONE>(a, s_item); item < a.nitems;
         item = next_item<ONE>(a, item, s_item)) {
        if constexpr (!ONE) load_desc(a, item, sdm, s_inst, cur_inst);
        const InstDesc& sd = desc_of<ONE>(a, sdm);
        if (member_done<ONE>(a, sd)) continue;   // block-uniform

        const int nx = sd.nx, ny = sd.ny, nz = sd.nz, pitch = sd.pitch;
        const bool px = sd.per_x, py = sd.per_y, pz = sd.per_z;
        const long long local = item - sd.item_begin;
        const int txi = (int)(local % sd.ntx);
        const int tyi = (int)((local / sd.ntx) % sd.nty);
        const int zc = (int)(local / ((long long)sd.ntx * sd.nty));
        const int x0 = txi * kTileQ * kVEC, y0 = tyi * TY;
        const int z0 = zc * sd.zchunk;
        if (!ONE && z0 >= nz) continue;   // no such item: the march ends on == z1
        const int z1 = min(z0 + sd.zchunk, nz);
        const int lin = sd.par ^ a.parity;
        const ST* const gin = reinterpret_cast<const ST*>(sd.base[lin][PASS == 1 ? 2 : 0]);
        ST* const gout = reinterpret_cast<ST*>(sd.base[lin ^ 1][0]);
        const long long fstride =
            S > 1 ? reinterpret_cast<const ST*>(sd.base[lin][1]) -
                        reinterpret_cast<const ST*>(sd.base[lin][0])
                  : 0;
        const long long plane = sd.plane;

        const int y = y0 - 1 + t.r;                   // global row of the position
        const int xs = x0 - kVEC + t.v * kVEC;        // global x of its first element
        const bool stores = inner && y < ny && xs < nx;
        const XSides sides(t, inner, xs, x0, nx, px);
        const unsigned xyf = xy_faces(xs, y, nx, ny);
        const bool src_col = sd.src_s >= 0 && (py ? wrapi(y, ny) : y) == sd.src_y;
        const bool elems = sd.wrap_elems;
        // k6: D dt / (6 h^2) per species; PASS 1: p[2] / 6 (mu); PASS 2:
        // k6[2] = p[1] / 6 (the mobility term of c)
        float k6[S];
#pragma unroll
        for (int s = 0; s < S; ++s) k6[s] = __fdiv_rn(sd.kx[s], 6.0f);
        if constexpr (PASS == 1) k6[0] = __fdiv_rn(sd.p[2], 6.0f);
        if constexpr (PASS == 2) k6[2] = __fdiv_rn(sd.p[1], 6.0f);
        if constexpr (ONE) chain_wait();   // nothing above reads what a launch writes
        float cy = 0.0f, cz = 0.0f;                   // 3-D wind
        if constexpr (W3 && PASS == 0) wind3d(sd, lin, local, cy, cz);
        // what the thread copies of every plane: its own vector, offset ``go``
        // of a plane (see own_offset), or for the halo warp three vectors a
        // lane, described in shared memory
        unsigned go = kNone;
        if (inner) {
            const Fetch f = make_fetch_h<ST>(y, xs, nx, ny, pitch, px, py, 0);
            go = own_offset(f);
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int j = min(tid + 32 * k, ninner + TilePos::ring(TY) - 1);
                const TilePos h(j, TY);
                const Fetch f = make_fetch_h<ST>(y0 - 1 + h.r, x0 - kVEC + h.v * kVEC, nx, ny,
                                                 pitch, px, py,
                                                 kGuard19 + h.r * ROWB + h.v * kVEC * EB);
                if (RD_DBG_SHARED(hfetch + hl + 32 * k, 16, kSiteHaloDesc))
                    hfetch[hl + 32 * k] = make_int4(f.mode, (int)f.goff, f.soff, f.xs);
            }
            __syncwarp();
        }
        // from a vector's place in the state fields to that in mu
        auto mu_shift = [&](int vx) { return NS * SPB + ((vx - x0) + kVEC) * (4 - EB); };

        // planes z0-1 .. z1 are copied; the next one to slot_ld
        PlaneFeed feed(z0 - 1, nz, pz);
        const int slot_end = own0 + RING * SLOTB;
        int slot_ld = own0;
        // vector o of the plane at goff, to d (mu: dm)
        auto copy = [&](long long goff, unsigned o, unsigned char* d, unsigned char* dm, bool ok) {
            goff += (unsigned long long)o * kVEC;
            const ST* const g = gin + goff;
#pragma unroll
            for (int s = 0; s < NS; ++s)
                Store<ST>::cp_async_if(
                    reinterpret_cast<ST*>(d + s * SPB), g + s * fstride,
                    ok && RD_DBG_GLOBAL(sd, g + s * fstride, 4 * (int)sizeof(ST), kSiteCopySrc));
            if constexpr (MUF) {
                const float* const gm = sd.mu + goff;
                Store<float>::cp_async_if(reinterpret_cast<float*>(dm), gm,
                                          ok && RD_DBG_GLOBAL(sd, gm, 16, kSiteMu));
            }
        };
        auto copy_elems = [&](long long goff, Fetch f, unsigned char* d) {
            fetch_elems<ST, NS>(f, d, SPB, gin + goff, fstride, nx, sd);
            if constexpr (MUF) {
                f.soff += mu_shift(f.xs);
                fetch_elems<float, 1>(f, d, 0, sd.mu + goff, 0, nx, sd);
            }
        };
        auto issue = [&]() {
            if (feed.n <= z1) {
                const long long goff = (long long)feed.plane() * plane;
                unsigned char* const d = smem + slot_ld;
                if (inner_warp) {
                    copy(goff, go, d, d + mu_own, go < kElems);
                } else {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const int4 h = hfetch[hl + 32 * k];
                        unsigned char* const dk = d - own0 + h.z;
                        copy(goff, (unsigned)h.y, dk, dk + mu_shift(h.w), h.x == 1);
                    }
                }
                if (elems) {   // periodic x, nx not a multiple of 4
                    if (go == kElems)
                        copy_elems(goff, Fetch{2, row_offset(y, ny, pitch, py), 0, xs}, d);
                    if (!inner_warp)
                        for (int k = 0; k < 3; ++k) {
                            const int4 h = hfetch[hl + 32 * k];
                            copy_elems(goff, Fetch{h.x, (unsigned)h.y, h.z, h.w}, d - own0);
                        }
                }
            }
            feed.next();
            slot_ld += SLOTB;
            if (slot_ld == slot_end) slot_ld = own0;
            cp_async_commit();
        };
        // plane sums of field i of the slot whose own vector is at ``p``
        auto sums = [&](const unsigned char* p, int i, float(&c)[kVEC], float(&zs)[kVEC],
                        float(&ws)[kVEC]) {
            if (MUF && i == NSUM - 1) plane_sums19<float, ROWB>(sides, p + mu_own, c, zs, ws);
            else plane_sums19<ST, ROWB>(sides, p + i * SPB, c, zs, ws);
        };
#pragma unroll 1
        for (int j = 0; j < P; ++j) issue();

        ST* gst = gout + (long long)z0 * plane + (long long)y * pitch + xs;
        float* gmu_st = nullptr;
        if constexpr (PASS == 1) gmu_st = sd.mu + (long long)z0 * plane + (long long)y * pitch + xs;
        int slot = own0;                              // ring slot of plane q - 1
        auto next_slot = [&](int x) {
            x += SLOTB;
            return x == slot_end ? own0 : x;
        };
        // three sets each of the sums and own vectors, roles rotating; CC: the
        // own c of PASS 2
        float ZA[NSUM][kVEC], ZB[NSUM][kVEC], ZC[NSUM][kVEC];
        float WA[NSUM][kVEC], WB[NSUM][kVEC], WC[NSUM][kVEC];
        float CA[NSUM][kVEC], CB[NSUM][kVEC], CC[NSUM][kVEC];
        float DA[kVEC], DB[kVEC], DC[kVEC];
        // the step for plane q: sums of planes q - 1 and q in zm and z0, w0,
        // own vectors of planes q - 1 and q in cm and c0; those of plane
        // q + 1 are formed here
        auto body = [&](int q, float(&zm)[NSUM][kVEC], float(&zq)[NSUM][kVEC],
                        float(&zp)[NSUM][kVEC], float(&wq)[NSUM][kVEC], float(&wp)[NSUM][kVEC],
                        float(&cm)[NSUM][kVEC], float(&c0)[NSUM][kVEC], float(&cp)[NSUM][kVEC],
                        float(&dq)[kVEC], float(&dp)[kVEC]) {
            // planes through q + 1 must have landed: of those issued, through
            // q + P - 2, all but the newest P - 3
            cp_async_wait<P - 3>();
            cta_barrier(blockDim.x);
            const int s0 = next_slot(slot);
            const unsigned char* const p0 = smem + s0;
            {
                const unsigned char* const p1 = smem + next_slot(s0);
                if constexpr (PASS == 2) lds_vec<ST>(p1 + 2 * SPB, dp);
                float lap6[NSUM][kVEC];   // 6 h^2 Lap of the fields on plane q
#pragma unroll
                for (int i = 0; i < NSUM; ++i) {
                    sums(p1, i, cp[i], zp[i], wp[i]);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        set_pair(lap6[i], h,
                                 vfma(vset<float2>(-24.0f), pair_of(c0[i], h),
                                      vadd(vadd(pair_of(zm[i], h), pair_of(zp[i], h)),
                                           pair_of(wq[i], h))));
                }
                if constexpr (PASS == 1) {
                    // mu = g(c) - (p[2] / 6) 6 h^2 Lap c
                    float mu[kVEC];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        set_pair(mu, h, vfma(vset<float2>(-k6[0]), pair_of(lap6[0], h),
                                             M::g(sd, pair_of(c0[0], h))));
                    if (stores && RD_DBG_GLOBAL(sd, gmu_st, 16, kSiteMu))
                        Store<float>::store(gmu_st, mu);
                    gmu_st += plane;
                } else {
                    // state of plane q: a, b (and every PASS 0 species) from
                    // the summed fields, c of PASS 2 from its own vector
                    float cen[S][kVEC], inc[S][kVEC];
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int i = 0; i < kVEC; ++i)
                            cen[s][i] = (PASS == 2 && s == 2) ? dq[i] : c0[s < NSUM ? s : 0][i];
                    react4<M>(sd, cen, inc);
                    if (W3 && (cy != 0.0f || cz != 0.0f)) {
                        // upwind along y and z (3-D wind): y neighbours of
                        // plane q, z neighbours the thread's own vectors
#pragma unroll
                        for (int s = 0; s < S; ++s) {
                            float ym[kVEC], yp[kVEC];
                            lds_vec<ST>(p0 + s * SPB - ROWB, ym);
                            lds_vec<ST>(p0 + s * SPB + ROWB, yp);
                            upwind_axis(cy, cen[s], ym, yp, inc[s]);
                            upwind_axis(cz, cen[s], cm[s < NSUM ? s : 0], cp[s < NSUM ? s : 0],
                                        inc[s]);
                        }
                    }
                    const float cx = PLAIN ? 0.0f : courant_at(sd, sd.courant, q);
                    const bool src_here = src_col && q == sd.src_z;
                    const unsigned faces = xyf | z_faces(q, nz);
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        float o[kVEC];
                        // PASS 2, c: the Laplacian is that of mu (summed field 2)
                        const float(&ls)[kVEC] = lap6[(PASS == 2 && s == 2) ? 2 : (s < NSUM ? s : 0)];
                        float left = 0.0f, right = 0.0f;
                        if (!PLAIN && cx != 0.0f) {
                            const unsigned char* ps = p0 + s * SPB;
                            left = lds_one<ST>(ps + sides.lcell * EB);
                            // (a face inside the vector: cen holds the ghost)
                            right = lds_one<ST>(ps + sides.rcell * EB);
                        }
                        species19<PLAIN>(sd, s, k6[s], cen[s], ls, inc[s], cx, left, right,
                                         src_here, px, xs, o);
                        if constexpr (!PLAIN) held_layers_at(sd, s, faces, xs, y, q, o);
                        if (stores && RD_DBG_GLOBAL(sd, gst + s * fstride, 4 * (int)sizeof(ST),
                                                    kSiteStateStore))
                            Store<ST>::store(gst + s * fstride, o);
                    }
                    gst += plane;
                }
            }
            // refills the slot of plane q - 1; last, behind the step's own loads
            issue();
            slot = s0;
        };
        // the sums of the first two planes, formed before the first barrier of
        // the march, after which their slots are refilled
        cp_async_wait<P - 2>();
        cta_barrier(blockDim.x);
        if (inner_warp) {
            float w[kVEC];
#pragma unroll
            for (int i = 0; i < NSUM; ++i) {
                sums(smem + slot, i, CA[i], ZA[i], w);
                sums(smem + next_slot(slot), i, CB[i], ZB[i], WA[i]);
            }
            if constexpr (PASS == 2) lds_vec<ST>(smem + next_slot(slot) + 2 * SPB, DA);
            for (int q = z0;;) {
                body(q, ZA, ZB, ZC, WA, WB, CA, CB, CC, DA, DB);
                if (++q == z1) break;
                body(q, ZB, ZC, ZA, WB, WC, CB, CC, CA, DB, DC);
                if (++q == z1) break;
                body(q, ZC, ZA, ZB, WC, WA, CC, CA, CB, DC, DA);
                if (++q == z1) break;
            }
        } else {   // the halo warp only copies
#pragma unroll 1
            for (int q = z0; q < z1; ++q) {
                cp_async_wait<P - 3>();
                cta_barrier(blockDim.x);
                issue();
            }
        }
        if (ONE && item + gridDim.x >= a.nitems) chain_release();   // the last item
        cp_async_wait<0>();
        __syncthreads();
    }
}

// Launch helper used by the per-model translation units: even tile heights
// (16 TY compute threads, then a whole halo warp); single instances (the
// descriptor in the kernel parameters) or batches (a device array of
// descriptors).
template <class M, class ST, int PASS>
cudaError_t launch19_pass(const LaunchArgs& a, int grid, size_t smem, cudaStream_t st, int* occ) {
    if ((a.ty & 1) || a.ty < 2) return cudaErrorInvalidValue;
    void (*k)(const LaunchArgs);
    const bool w3 = PASS == 0 && !a.plain && a.wind3;
    if (a.use_one)
        k = a.plain ? rd_march19_kernel<M, ST, true, true, PASS>
            : w3    ? rd_march19_kernel<M, ST, true, false, PASS, PASS == 0>
                    : rd_march19_kernel<M, ST, true, false, PASS>;
    else
        k = a.plain ? rd_march19_kernel<M, ST, false, true, PASS>
            : w3    ? rd_march19_kernel<M, ST, false, false, PASS, PASS == 0>
                    : rd_march19_kernel<M, ST, false, false, PASS>;
    static size_t configured[6] = {0, 0, 0, 0, 0, 0};
    size_t& conf = configured[(a.plain ? 1 : w3 ? 2 : 0) + (a.use_one ? 3 : 0)];
    if (smem > conf) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        conf = smem;
    }
    const int threads = Layout19<M, ST, PASS>::threads(a.ty);
    if (threads > kMaxThreads) return cudaErrorInvalidConfiguration;
    if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, threads, smem);
    return launch_chained(k, a, grid, threads, smem, st);
}

template <class M>
cudaError_t launch19_model(int storage, const LaunchArgs& a, int grid, size_t smem,
                           cudaStream_t st, int* occ) {
    if (storage == RD_STORE_F32) return launch19_pass<M, float, 0>(a, grid, smem, st, occ);
    if (storage == RD_STORE_BF16)
        return launch19_pass<M, __nv_bfloat16, 0>(a, grid, smem, st, occ);
    return cudaErrorInvalidValue;
}

// The two launches of a Cahn-Hilliard step: pass 1 (mu), pass 2 (update).
// ``smem`` is pass 2's size; pass 1 takes the smaller ring of its own layout.
template <class M>
cudaError_t launch19_ch_model(int storage, int pass, const LaunchArgs& a, int grid, size_t smem,
                              cudaStream_t st, int* occ) {
    if (storage == RD_STORE_F32)
        return pass == 1 ? launch19_pass<M, float, 1>(a, grid, Layout19<M, float, 1>::total(a.ty),
                                                      st, occ)
                         : launch19_pass<M, float, 2>(a, grid, smem, st, occ);
    if (storage == RD_STORE_BF16)
        return pass == 1 ? launch19_pass<M, __nv_bfloat16, 1>(
                               a, grid, Layout19<M, __nv_bfloat16, 1>::total(a.ty), st, occ)
                         : launch19_pass<M, __nv_bfloat16, 2>(a, grid, smem, st, occ);
    return cudaErrorInvalidValue;
}

}  // namespace rdk
