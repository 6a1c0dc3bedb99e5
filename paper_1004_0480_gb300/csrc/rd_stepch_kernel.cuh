// rd_stepch_kernel.cuh -- the one-step kernel of the models with a
// Cahn-Hilliard species (7-point stencil), included from rd_step_kernel.cuh
// after rd_march_kernel.cuh, whose layout it takes.
#pragma once

namespace rdk {

// The T = 1 path of the models with a Cahn-Hilliard species c (the front
// model a + b -> c, and the phase separation of Table 1, row 3): the two-step
// march with mu in the place of level 1.  At the step for plane e a thread
// forms mu of plane e at its position of the widened tile (halo warps do only
// that), and the inner threads the new state of plane e - 1.  Rows and planes
// beyond a zero-flux y or z face are mirror images, so mu computed at a ghost
// cell equals mu at the face cell (the pair along the mirrored axis holds the
// same two values swapped) -- the paper's "Laplacian, boundary rule,
// Laplacian"; along x the face cell is its own neighbour, for c and for mu.
//
// A thread carries its own a and b of planes e - 2 .. e, c of e - 1 .. e + 1
// and mu of e - 2 .. e in register sets whose roles rotate.  State planes
// arrive in a ring of 6, three ahead: at step e the neighbours of a and b in
// plane e - 1 and of c in plane e are read, and the slot of plane e - 2, last
// read at step e - 1, is refilled.  mu passes through 2 slots: the one written
// at step e held plane e - 2, last read at step e - 1.  One barrier per plane.
// The rows at distance two hold c only.
template <class ST> struct LayoutCH {
    static constexpr int S = 3;
    using RM = RowMap<S, ST>;
    using RMU = RowMap<1, float>;
    static constexpr int RING = 6;        // planes e - 1 .. e + 4
    static constexpr int P = RING - 1;    // planes issued ahead of plane e - 2
    // registers a thread may take; front 192^3 FP32, GLUPS at the best
    // tiling when the budget was chosen (210 now): 200 (128), 208 (112), 158
    // (96); the kernel before it (mirrored ghosts element by element, loads
    // with a 4-way conflict): 188; eight uneven fronts batched 145 against 113
    static constexpr int regs(bool lean) { return lean && sizeof(ST) == 4 ? 112 : 128; }
    __host__ __device__ static size_t state_bytes(int ty) {
        return (size_t)RING * RM::plane_bytes(ty + 4);
    }
    __host__ __device__ static size_t total(int ty) {
        return state_bytes(ty) + (size_t)2 * RMU::plane_bytes(ty + 2);
    }
    // whole warps: the inner positions, then the halo ring (its last warp
    // repeats the last position, writing the same values); at an odd height
    // one warp holds both
    __host__ __device__ static int threads(int ty) { return (kNQ * (ty + 2) + 31) / 32 * 32; }
};

// PLAIN: no point source or wind and isotropic D for a and b (held layers
// are still applied); the update of a and b then needs no per-plane tests.
template <class MC, class ST, bool ONE, bool PLAIN>
__global__ void __maxnreg__((LayoutCH<ST>::regs(PLAIN)))
rd_marchch_kernel(const __grid_constant__ LaunchArgs a) {
    using LY = LayoutCH<ST>;
    using RM = typename LY::RM;
    using RMU = typename LY::RMU;
    constexpr int S = 3;
    constexpr int P = LY::P;
    constexpr int RING = LY::RING;
    constexpr int EB = (int)sizeof(ST);
    constexpr unsigned FULL = 0xffffffffu;

    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ InstDesc sdm;
    __shared__ int s_inst;
    __shared__ long long s_item;

    const int tid = threadIdx.x;
    const int TY = a.ty;
    const int SLOTB = RM::plane_bytes(TY + 4);
    const int SLOTM = RMU::plane_bytes(TY + 2);
    const int ninner = kTileQ * TY;
    const TilePos t(min(tid, ninner + TilePos::ring(TY) - 1), TY);
    const int hl = tid - ninner;                             // >= 0: halo thread
    const bool inner = hl < 0;
    const bool update_warp = __any_sync(FULL, inner);
    const bool halo_warp = __any_sync(FULL, !inner);
    // byte offsets of the own vector in slot 0 of the state and mu rings
    const int own0 = kVEC * EB + (t.r + 1) * RM::ROWB + t.v * kVEC * EB;
    const int ownm = (int)LY::state_bytes(TY) + (kVEC + t.v * kVEC) * 4 + t.r * RMU::ROWB;

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
        const ST* const gin = reinterpret_cast<const ST*>(sd.base[lin][0]);
        ST* const gout = reinterpret_cast<ST*>(sd.base[lin ^ 1][0]);
        const long long fstride = reinterpret_cast<const ST*>(sd.base[lin][1]) - gin;
        const long long plane = sd.plane;

        const int y = y0 - 1 + t.r;                   // global row of the position
        const int xs = x0 - kVEC + t.v * kVEC;        // global x of its first element
        const bool stores = inner && y < ny && xs < nx;
        const XSides sides(t, inner, xs, x0, nx, px);
        const unsigned xyf = xy_faces(xs, y, nx, ny);
        const bool src_col = sd.src_s >= 0 && (py ? wrapi(y, ny) : y) == sd.src_y;
        const bool elems = sd.wrap_elems;
        // own state vector, and (first 2 x 18 halo threads) c of the outer rows
        const Fetch fo = make_fetch_h<ST>(y, xs, nx, ny, pitch, px, py, 0);
        Fetch fx{0, 0, 0, 0};
        if (hl >= 0 && hl < 2 * kNQ)
            fx = make_fetch_h<ST>(t.r ? y + 1 : y - 1, xs, nx, ny, pitch, px, py,
                                  (t.r ? RM::ROWB : -RM::ROWB) + 2 * RM::SPB);

        if constexpr (ONE) chain_wait();   // nothing above reads what a launch writes
        // planes z0-2 .. z1+1 are copied; the next one to slot_ld
        PlaneFeed feed(z0 - 2, nz, pz);
        const int slot_end = own0 + RING * SLOTB;
        int slot_ld = own0;
        auto issue = [&]() {
            if (feed.n <= z1 + 1) {
                const ST* g = gin + (long long)feed.plane() * plane;
                unsigned char* const d = smem + slot_ld;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const ST* gs = vec_at(g, fo.goff) + s * fstride;
                    const int ok = fo.mode == 1 &&
                                   RD_DBG_GLOBAL(sd, gs, 4 * (int)sizeof(ST), kSiteCopySrc);
                    Store<ST>::cp_async_if(reinterpret_cast<ST*>(d + s * RM::SPB), gs, ok);
                }
                if (halo_warp) {
                    const ST* gs = vec_at(g, fx.goff) + 2 * fstride;
                    const int ok = fx.mode == 1 &&
                                   RD_DBG_GLOBAL(sd, gs, 4 * (int)sizeof(ST), kSiteCopySrc);
                    Store<ST>::cp_async_if(reinterpret_cast<ST*>(d + fx.soff), gs, ok);
                }
                if (elems) {   // periodic x, nx not a multiple of 4
                    fetch_elems<ST, S>(fo, d, RM::SPB, g, fstride, nx, sd);
                    fetch_elems<ST, 1>(fx, d, 0, g + 2 * fstride, 0, nx, sd);
                }
            }
            feed.next();
            slot_ld += SLOTB;
            if (slot_ld == slot_end) slot_ld = own0;
            cp_async_commit();
        };
#pragma unroll 1
        for (int j = 0; j < P; ++j) issue();

        ST* gst = gout + (long long)z0 * plane + (long long)y * pitch + xs;
        const int first = z0 - 1;
        int slot = own0;                              // ring slot of plane e - 1
        int parm = 0;                                 // mu slot of plane e - 1
        auto next_slot = [&](int x) {
            x += SLOTB;
            return x == slot_end ? own0 : x;
        };
        // own a, b; c; mu of three successive planes, roles rotating
        float AA[2][kVEC], AB[2][kVEC], AC[2][kVEC];
        float CA[1][kVEC], CB[1][kVEC], CC[1][kVEC];
        float MA[1][kVEC], MB[1][kVEC], MX[1][kVEC];
        // the step for plane e: a, b of planes e - 2, e - 1, e in am, a0, ap,
        // c of e - 1, e, e + 1 in cm, c0, cp, mu of e - 2, e - 1, e in mm,
        // m0, mp
        auto body = [&](int e, float(&am)[2][kVEC], float(&a0)[2][kVEC], float(&ap)[2][kVEC],
                        float(&cm)[1][kVEC], float(&c0)[1][kVEC], float(&cp)[1][kVEC],
                        float(&mm)[1][kVEC], float(&m0)[1][kVEC], float(&mp)[1][kVEC]) {
            // planes through e + 1 must have landed: of those issued, through
            // e + P - 2, all but the newest P - 3
            cp_async_wait<P - 3>();
            __syncthreads();
            const int s1 = next_slot(slot);
            const int s2 = next_slot(s1);
            if (e == first) {
                lds_vec<ST>(smem + slot + 2 * RM::SPB, cm[0]);
                lds_vec<ST>(smem + s1 + 2 * RM::SPB, c0[0]);
                sides.set_ghost(c0);
            }
            lds_vec<ST>(smem + s2 + 2 * RM::SPB, cp[0]);
            sides.set_ghost(cp);
#pragma unroll
            for (int s = 0; s < 2; ++s) lds_vec<ST>(smem + s1 + s * RM::SPB, ap[s]);
            sides.set_ghost(ap);
            issue();   // refills the slot of plane e - 2
            {
                // mu of plane e
                const unsigned char* const pc = smem + s1 + 2 * RM::SPB;
                float xm[kVEC], xp[kVEC], ym[kVEC], yp[kVEC];
                lds_vec<ST>(pc - RM::ROWB, ym);
                lds_vec<ST>(pc + RM::ROWB, yp);
                sides.get<ST>(c0[0], pc, xm, xp);
                mu4<MC>(sd, c0[0], xm, xp, ym, yp, cm[0], cp[0], mp[0]);
                Store<float>::store(reinterpret_cast<float*>(smem + ownm + (parm ^ SLOTM)), mp[0]);
                sides.set_ghost(mp);
            }
            if (e > z0 && update_warp) {
                // the new state of plane e - 1
                const int q = e - 1;
                const unsigned faces = xyf | z_faces(q, nz);
                float cen[S][kVEC], inc[S][kVEC];
#pragma unroll
                for (int i = 0; i < kVEC; ++i) {
                    cen[0][i] = a0[0][i];
                    cen[1][i] = a0[1][i];
                    cen[2][i] = cm[0][i];
                }
                react4<MC>(sd, cen, inc);
                const float cx = PLAIN ? 0.0f : courant_at(sd, sd.courant, q);
                const bool src_here = src_col && q == sd.src_z;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const unsigned char* const ps = smem + slot + s * RM::SPB;
                    float xm[kVEC], xp[kVEC], ym[kVEC], yp[kVEC], o[kVEC];
                    lds_vec<ST>(ps - RM::ROWB, ym);
                    lds_vec<ST>(ps + RM::ROWB, yp);
                    sides.get<ST>(cen[s], ps, xm, xp);
                    if constexpr (PLAIN)
                        euler4_iso(cen[s], xm, xp, ym, yp, am[s], ap[s], sd.kx[s], inc[s], o);
                    else
                        species_core(sd, s, cen[s], xm, xp, ym, yp, am[s], ap[s], inc[s], cx,
                                     src_here, px, xs, o);
                    held_layers_at(sd, s, faces, xs, y, q, o);
                    if (stores &&
                        RD_DBG_GLOBAL(sd, gst + s * fstride, 4 * (int)sizeof(ST), kSiteStateStore))
                        Store<ST>::store(gst + s * fstride, o);
                }
                {
                    // c += dt M / h^2 * (7-point Laplacian of mu)
                    const unsigned char* const pm = smem + ownm + parm;
                    float xm[kVEC], xp[kVEC], ym[kVEC], yp[kVEC], o[kVEC];
                    Store<float>::load(reinterpret_cast<const float*>(pm - RMU::ROWB), ym);
                    Store<float>::load(reinterpret_cast<const float*>(pm + RMU::ROWB), yp);
                    sides.get<float>(m0[0], pm, xm, xp);
                    euler4_ch(sd.p[1], cen[2], m0[0], xm, xp, ym, yp, mm[0], mp[0], inc[2], o);
                    held_layers_at(sd, 2, faces, xs, y, q, o);
                    if (stores &&
                        RD_DBG_GLOBAL(sd, gst + 2 * fstride, 4 * (int)sizeof(ST), kSiteStateStore))
                        Store<ST>::store(gst + 2 * fstride, o);
                }
            }
            if (e > z0) gst += plane;
            parm ^= SLOTM;
            slot = s1;
        };
        for (int e = first;;) {
            body(e, AA, AB, AC, CA, CB, CC, MA, MB, MX);
            if (++e == z1 + 1) break;
            body(e, AB, AC, AA, CB, CC, CA, MB, MX, MA);
            if (++e == z1 + 1) break;
            body(e, AC, AA, AB, CC, CA, CB, MX, MA, MB);
            if (++e == z1 + 1) break;
        }
        if (ONE && item + gridDim.x >= a.nitems) chain_release();   // the last item
        cp_async_wait<0>();
        __syncthreads();
    }
}

}  // namespace rdk
