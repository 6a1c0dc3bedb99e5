// rd_march_kernel.cuh -- one or two steps per launch, 7-point stencil, models
// without Cahn-Hilliard (sm_103a); included from rd_step_kernel.cuh.
//
// What bounds one step per launch on large grids is HBM: every step reads
// and writes the whole state.  With T = 2 a launch reads the state once,
// keeps the state after the first step (level 1) on chip and writes the
// state after the second, so the traffic per step halves, and so do the
// launches, which bound small grids.  What bounds the march itself is
// latency and instruction issue (some 16 to 24 warps fit on an SM), so its
// layout is chosen to spend few instructions and registers per cell:
//
//  * T = 2: one thread per 4-cell vector of a 64 x TY tile widened by one
//    vector in x and one row in y.  The 16 x TY inner positions come first
//    (whole warps: TY is even), the halo ring last, so halo warps compute
//    level 1 only.  At the step for plane e a thread advances level 0 of
//    plane e at its position, and the inner threads level 1 of plane e - 1.
//    T = 1: the inner threads, and one halo warp that only copies.
//  * The z neighbours at both levels are a thread's own vectors, carried in
//    registers down the march; three sets change roles from plane to plane,
//    written out three times, so that no register moves.  Only x and y
//    neighbours pass through shared memory: level 0 of plane e (a ring of 5
//    planes, filled by 16-byte cp.async three planes ahead) and level 1 of
//    plane e - 1 (2 slots).
//  * An inner thread takes the x neighbours beside its vector from the
//    adjacent lanes by warp shuffle; the lanes at a tile row's ends, and at a
//    zero-flux x face, read shared memory instead (their own cell at a face):
//    predicated loads, no branch and no 4-way bank conflict.
//  * One barrier per plane.  The copy of plane e + 4 is issued after the
//    barrier of step e into the slot of plane e - 1, whose neighbours were
//    last read at step e - 1.  The level-1 slot written at step e held plane
//    e - 2, last read at step e - 1.
//
// Measured at 2 steps per launch against the one-step kernel before it
// (4-cell vectors, one halo warp, scalar arithmetic), best tilings: 256^3
// Brusselator FP32 376 -> 504 GLUPS, 512^3 diffusion 814 -> 1124, 192^3
// Turing 294 -> 454, a 97 x 65 x 50 zero-flux Brusselator 32 -> 120; at one
// step per launch 376 -> 386 (HBM), BF16 428 -> 455.
//
// Boundary rules: rows and planes beyond a zero-flux y or z face are copied
// in by mirror extension to distance T, so level 1 evaluated on a ghost
// equals level 1 of the face cell bit for bit (the pair along the mirrored
// axis holds the same two values swapped; at T = 2 the wind blows along x).
// Along x nothing is computed beyond a face: the face cell is its own
// neighbour.  Level 1 is rounded to the state's type and takes its held
// layers, and both levels use the per-cell functions of rd_step_kernel.cuh,
// so a launch equals two one-step launches bit for bit.
#pragma once

namespace rdk {

// Shared-memory rows of the march kernels below hold every species of a
// row side by side, kRW elements each, so that a thread reaches all it reads
// in a plane from one address with compile-time offsets.  RowMap<S, ST>: byte
// strides of a row and of a species within it.
template <int S, class ST> struct RowMap {
    static constexpr int SPB = kRW * (int)sizeof(ST);
    static constexpr int ROWB = S * SPB;
    // bytes of ``rows`` rows, with a guard vector at both ends
    __host__ __device__ static constexpr int plane_bytes(int rows) {
        return rows * ROWB + 2 * kVEC * (int)sizeof(ST);
    }
};

// l / r = the elements at shared addresses pl / pr where ql / qr hold (no
// branch)
template <class ST>
__device__ __forceinline__ void lds_sides_if(float& l, float& r, const void* pl, const void* pr,
                                             int ql, int qr);
template <>
__device__ __forceinline__ void lds_sides_if<float>(float& l, float& r, const void* pl,
                                                    const void* pr, int ql, int qr) {
    if (ql && !RD_DBG_SHARED(pl, 4, kSiteSharedLoad)) return;
    if (qr && !RD_DBG_SHARED(pr, 4, kSiteSharedLoad)) return;
    asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
                 " @p ld.shared.f32 %0, [%2];\n @q ld.shared.f32 %1, [%3];\n}\n"
                 : "+f"(l), "+f"(r)
                 : "r"(static_cast<unsigned>(__cvta_generic_to_shared(pl))),
                   "r"(static_cast<unsigned>(__cvta_generic_to_shared(pr))), "r"(ql), "r"(qr)
                 : "memory");
}
template <>
__device__ __forceinline__ void lds_sides_if<__nv_bfloat16>(float& l, float& r, const void* pl,
                                                            const void* pr, int ql, int qr) {
    if (ql && !RD_DBG_SHARED(pl, 2, kSiteSharedLoad)) return;
    if (qr && !RD_DBG_SHARED(pr, 2, kSiteSharedLoad)) return;
    asm volatile("{\n .reg .pred p, q;\n .reg .b16 h, k;\n setp.ne.b32 p, %4, 0;\n"
                 " setp.ne.b32 q, %5, 0;\n"
                 " @p ld.shared.b16 h, [%2];\n @q ld.shared.b16 k, [%3];\n"
                 " @p mov.b32 %0, {0, h};\n @q mov.b32 %1, {0, k};\n}\n"
                 : "+f"(l), "+f"(r)
                 : "r"(static_cast<unsigned>(__cvta_generic_to_shared(pl))),
                   "r"(static_cast<unsigned>(__cvta_generic_to_shared(pr))), "r"(ql), "r"(qr)
                 : "memory");
}

template <class M, class ST, int T> struct LayoutM {
    static constexpr int S = M::S;
    using RM = RowMap<S, ST>;
    static constexpr int RING = 5;        // level-0 planes e .. e + 4
    static constexpr int P = 5;           // planes issued ahead of plane e - 1
    // Registers a thread may take.  The march is bound by latency (16 warps
    // on an SM at 128 registers), so what lets another CTA in pays for a few
    // spills.  Measured when the budgets were chosen (the kernel has gained a
    // few per cent since), GLUPS, at the best tiling of each:
    //   diffusion 512^3 FP32, T = 2: 933 (128) 935 (112) 986 (96) 1080 (80)
    //                         T = 1: 665 (96) 735 (80) 802 (64)
    //   Brusselator 256^3 FP32, T = 2: 433 (128) 427 (112) 478 (96) 401 (80)
    //                           T = 1: 366 (128) 371 (96) 387 (80) 291 (64)
    //   the same in BF16, T = 2: 441 (128) 362 (112) 312 (96)
    //                     T = 1: 457 (128) 451 (96) 401 (80) 296 (64)
    //   air 512 x 512 x 64 FP32, T = 1: 253 (128) 249 (112) 215 (96)
    // The general variants and batches take 16 more where that is below 128.
    static constexpr int regs(bool lean) {
        if (S == 3 || (S == 2 && sizeof(ST) == 2)) return 128;
        return (S == 2 ? (T == 2 ? 96 : 80) : (T == 2 ? 80 : 64)) + (lean ? 0 : 16);
    }
    __host__ __device__ static size_t ring_bytes(int ty) {
        return (size_t)RING * RM::plane_bytes(ty + 2 * T);
    }
    __host__ __device__ static size_t total(int ty) {
        return ring_bytes(ty) + (T == 2 ? (size_t)2 * RM::plane_bytes(ty + 2) : 0);
    }
    // whole warps.  T = 2: the inner positions, then the halo ring (its last
    // warp repeats the last position, writing the same values); T = 1: the
    // inner positions, then a halo warp that only copies
    __host__ __device__ static int threads(int ty) {
        return T == 2 ? (kNQ * (ty + 2) + 31) / 32 * 32 : kTileQ * ty + 32;
    }
};

// Mirror extension: -1-i for i < 0, 2n-1-i for i >= n; clamped so that
// positions outside the grid by more than n (never stored) stay in bounds.
__host__ __device__ __forceinline__ int mirror_index(int i, int n) {
    const int m = i < 0 ? -1 - i : (i >= n ? 2 * n - 1 - i : i);
    return min(max(m, 0), n - 1);
}

// Offset of the row that stands for row ``yrow`` within a plane, in vectors.
__host__ __device__ __forceinline__ unsigned row_offset(int yrow, int ny, int pitch, bool py) {
    return (unsigned)(py ? wrapi(yrow, ny) : mirror_index(yrow, ny)) * ((unsigned)pitch / kVEC);
}

// How one vector of a march is fetched: rows beyond a zero-flux y face are
// mirror images, vectors beyond a zero-flux x
// face are not fetched, and the last vector of a row that ends inside it is
// copied whole (its tail is the row's padding, never read).
template <class ST>
__host__ __device__ __forceinline__ Fetch make_fetch_h(int yrow, int xs, int nx, int ny, int pitch,
                                                      bool px, bool py, int soff_bytes) {
    Fetch f{0, 0, soff_bytes, xs};
    if (yrow > ny + 1 || xs > nx + 1) return f;          // feeds no stored cell
    const unsigned row = row_offset(yrow, ny, pitch, py);
    if (xs >= 0 && xs + kVEC <= nx) {
        f.mode = 1;
        f.goff = row + (unsigned)xs / kVEC;
    } else if (px) {
        const int xw = wrapi(xs, nx);
        if (xw % kVEC == 0 && xw + kVEC <= nx) { f.mode = 1; f.goff = row + (unsigned)xw / kVEC; }
        else { f.mode = 2; f.goff = row; }
    } else if (xs >= 0 && xs < nx) {
        f.mode = 1;
        f.goff = row + (unsigned)xs / kVEC;
    }
    return f;
}

// Element copies of a vector that wraps round a periodic x axis (mode 2).
template <class ST, int S>
__device__ __forceinline__ void fetch_elems(const Fetch& f, unsigned char* dst, int pe_bytes,
                                            const ST* gplane, long long fstride, int nx,
                                            const InstDesc& sd) {
    if (f.mode != 2) return;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        ST* d = reinterpret_cast<ST*>(dst + s * pe_bytes + f.soff);
#pragma unroll
        for (int e = 0; e < kVEC; ++e) {
            const ST* src = vec_at(gplane, f.goff) + s * fstride + wrapi(f.xs + e, nx);
            if (RD_DBG_GLOBAL(sd, src, (int)sizeof(ST), kSiteCopySrc))
                Store<ST>::cp_async_elem(d + e, src);
        }
    }
}

// Position (r, v) in the tile widened by one row and one vector on every
// side: row r - 1, vector v - 1.  The 16 x TY inner positions come first,
// then the halo ring: the row above, the row below, left and right of each
// row.
struct TilePos {
    int r, v;
    __device__ __forceinline__ static int ring(int TY) { return 2 * kNQ + 2 * TY; }
    __device__ __forceinline__ TilePos(int i, int TY) {
        const int j = i - kTileQ * TY;
        if (j < 0) {
            r = i / kTileQ + 1;
            v = i - (r - 1) * kTileQ + 1;
        } else if (j < kNQ) {
            r = 0;
            v = j;
        } else if (j < 2 * kNQ) {
            r = TY + 1;
            v = j - kNQ;
        } else {
            r = (j - 2 * kNQ) / 2 + 1;
            v = ((j - 2 * kNQ) & 1) ? kNQ - 1 : 0;
        }
    }
};

// The x neighbours beside a thread's vector: the adjacent lane's value, or
// (ends of a tile row, halo threads) the vector beside it in shared memory,
// or (zero-flux face on the vector's edge) the own face cell.
struct XSides {
    int llds, rlds;        // read shared memory instead of the adjacent lane
    int lcell, rcell;      // element read, from the own vector's first
    int cut;               // a zero-flux face inside the vector: the element
                           // past its last cell, else 0
    bool any_cut;          // block-uniform: the tile holds such a vector
    __device__ __forceinline__ XSides(const TilePos& t, bool inner, int xs, int x0, int nx,
                                       bool px) {
        const bool lface = !px && xs == 0, rface = !px && xs + kVEC == nx;
        llds = !inner || lface || t.v == 1;
        rlds = !inner || rface || t.v == kTileQ;
        lcell = lface ? 0 : -1;
        rcell = rface ? kVEC - 1 : kVEC;
        any_cut = !px && (nx & (kVEC - 1)) && x0 + (kTileQ + 1) * kVEC >= nx;
        cut = any_cut && xs < nx && nx < xs + kVEC ? nx - xs : 0;
    }
    // neighbours of the own vector c, which sits at ``p`` in shared memory;
    // called by whole warps
    template <class ST>
    __device__ __forceinline__ void get(const float (&c)[kVEC], const unsigned char* p,
                                        float (&xm)[kVEC], float (&xp)[kVEC]) const {
        constexpr unsigned FULL = 0xffffffffu;
        float left = __shfl_up_sync(FULL, c[kVEC - 1], 1);
        float right = __shfl_down_sync(FULL, c[0], 1);
        lds_sides_if<ST>(left, right, p + lcell * (int)sizeof(ST), p + rcell * (int)sizeof(ST),
                         llds, rlds);
#pragma unroll
        for (int e = 0; e < kVEC; ++e) {
            xm[e] = e ? c[e - 1] : left;
            xp[e] = (e < kVEC - 1) ? c[e + 1] : right;
        }
    }
    // the same for a vector and those in the rows above and below (u, d):
    // every shuffle first, then the predicated loads, which overwrite shuffled
    // values and would stall the next row's shuffle
    template <class ST, int ROWB>
    __device__ __forceinline__ void get3(const float (&c)[kVEC], const float (&u)[kVEC],
                                         const float (&d)[kVEC], const unsigned char* p,
                                         float (&l)[3], float (&r)[3]) const {
        constexpr unsigned FULL = 0xffffffffu;
        l[0] = __shfl_up_sync(FULL, c[kVEC - 1], 1);
        l[1] = __shfl_up_sync(FULL, u[kVEC - 1], 1);
        l[2] = __shfl_up_sync(FULL, d[kVEC - 1], 1);
        r[0] = __shfl_down_sync(FULL, c[0], 1);
        r[1] = __shfl_down_sync(FULL, u[0], 1);
        r[2] = __shfl_down_sync(FULL, d[0], 1);
        const unsigned char* const pl = p + lcell * (int)sizeof(ST);
        const unsigned char* const pr = p + rcell * (int)sizeof(ST);
        lds_sides_if<ST>(l[0], r[0], pl, pr, llds, rlds);
        lds_sides_if<ST>(l[1], r[1], pl - ROWB, pr - ROWB, llds, rlds);
        lds_sides_if<ST>(l[2], r[2], pl + ROWB, pr + ROWB, llds, rlds);
    }
    // the ghost beside a zero-flux face inside the vector, set to the face
    // cell in a thread's own copy of the vectors of one plane
    __device__ __forceinline__ void set_ghost1(float (&c)[kVEC]) const {
        if (!any_cut) return;
        asm volatile("");   // keep the branch: rarely taken, uniform
#pragma unroll
        for (int e = kVEC - 1; e > 0; --e) c[e] = e == cut ? c[e - 1] : c[e];
    }
    template <int S> __device__ __forceinline__ void set_ghost(float (&c)[S][kVEC]) const {
        if (!any_cut) return;
        asm volatile("");   // keep the branch: rarely taken, uniform
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int e = kVEC - 1; e > 0; --e) c[s][e] = e == cut ? c[s][e - 1] : c[s][e];
    }
};

// A barrier of the whole CTA (nthreads: its size) for warps that run their own
// loops: every warp passes it the same number of times, wherever in the code.
__device__ __forceinline__ void cta_barrier(int nthreads) {
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// The global plane that the next copy reads, walked up from plane z0 - h:
// wrapped (periodic z) or mirrored at zero-flux faces.
struct PlaneFeed {
    int n, zw, nz;
    bool pz;
    __device__ __forceinline__ PlaneFeed(int first, int nz_, bool pz_)
        : n(first), zw(pz_ ? wrapi(first, nz_) : first), nz(nz_), pz(pz_) {}
    __device__ __forceinline__ int plane() const { return pz ? zw : mirror_index(n, nz); }
    __device__ __forceinline__ void next() {
        ++n;
        ++zw;
        if (pz && zw == nz) zw = 0;
    }
};

// What a problem may have beside reactions and diffusion, so that the kernel
// tests for nothing else: kPlain: no held layer, point source or wind, every
// species isotropic; kWindX: no held layer, wind along +x or none, every
// species anisotropic (the air problem, 512 x 512 x 64: 249 GLUPS, 0.88 of
// the HBM copy rate, against 197 in the general variant); kWind3: the 3-D wind
// (upwind along y and z too; T = 1); kGeneral: anything else.
enum MarchVar { kGeneral, kPlain, kWind3, kWindX };

template <class M, class ST, int T, bool ONE, int VAR>
__global__ void __maxnreg__((LayoutM<M, ST, T>::regs(ONE && VAR == kPlain)))
rd_march_kernel(const __grid_constant__ LaunchArgs a) {
    static_assert(T == 1 || T == 2, "one or two steps per launch");
    static_assert(VAR != kWindX || T == 1, "the Courant number is read one plane ahead");
    constexpr bool PLAIN = VAR == kPlain;
    constexpr bool W3 = VAR == kWind3;
    static_assert(!W3 || T == 1, "the 3-D wind steps once per launch");
    using LY = LayoutM<M, ST, T>;
    using RM = typename LY::RM;
    constexpr int S = M::S;
    constexpr int P = LY::P;
    constexpr int RING = LY::RING;
    constexpr int EB = (int)sizeof(ST);
    constexpr int NF = T == 2 ? 2 : 3;     // vectors a halo thread fetches
    constexpr unsigned FULL = 0xffffffffu;

    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ InstDesc sdm;
    __shared__ int s_inst;
    __shared__ long long s_item;

    const int tid = threadIdx.x;
    const int TY = a.ty;
    const int SLOTB = RM::plane_bytes(TY + 2 * T);           // level 0
    const int SLOTB1 = RM::plane_bytes(TY + 2);              // level 1
    const int ninner = kTileQ * TY;
    // halo threads: tile positions past the inner ones (T = 2; the last warp
    // repeats the last one); T = 1: a halo thread has none, its first fetch's
    // stands in
    const TilePos t(T == 2 ? min(tid, ninner + TilePos::ring(TY) - 1) : tid, TY);
    const int hl = tid - ninner;                             // >= 0: halo thread
    const bool inner = hl < 0;
    // TY is even: the inner threads are whole warps
    const bool inner_warp = __all_sync(FULL, inner);
    // byte offsets of the own vector in slot 0 of either ring
    const int own0 = kVEC * EB + (t.r + T - 1) * RM::ROWB + t.v * kVEC * EB;
    const int own1 = (int)LY::ring_bytes(TY) + kVEC * EB + t.r * RM::ROWB + t.v * kVEC * EB;

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
        const long long fstride = S > 1 ? reinterpret_cast<const ST*>(sd.base[lin][1]) - gin : 0;
        const long long plane = sd.plane;

        const int y = y0 - 1 + t.r;                   // global row of the position
        const int xs = x0 - kVEC + t.v * kVEC;        // global x of its first element
        const int yw = py ? wrapi(y, ny) : mirror_index(y, ny);
        const bool stores = inner && y < ny && xs < nx;
        const XSides sides(t, inner, xs, x0, nx, px);
        const unsigned xyf = xy_faces(xs, y, nx, ny);
        const bool src_col = sd.src_s >= 0 && yw == sd.src_y;
        const bool elems = sd.wrap_elems;
        if constexpr (ONE) chain_wait();   // nothing above reads what a launch writes
        float cy = 0.0f, cz = 0.0f;                   // 3-D wind
        if constexpr (W3) wind3d(sd, lin, local, cy, cz);
        // what the thread copies of every plane, offsets from its own vector:
        // its own vector, and for halo threads (T = 2) a vector of the rows
        // outside the halo ring or (T = 1) three vectors of the ring
        Fetch f[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) f[k] = Fetch{0, 0, 0, 0};
        if (T == 2 || inner) f[0] = make_fetch_h<ST>(y, xs, nx, ny, pitch, px, py, 0);
        if (!inner) {
            if constexpr (T == 2) {
                if (hl < 2 * kNQ)
                    f[1] = make_fetch_h<ST>(t.r ? y + 1 : y - 1, xs, nx, ny, pitch, px, py,
                                            t.r ? RM::ROWB : -RM::ROWB);
            } else {
#pragma unroll
                for (int k = 0; k < NF; ++k)
                    if (hl + 32 * k < TilePos::ring(TY)) {
                        const TilePos h(tid + 32 * k, TY);
                        f[k] = make_fetch_h<ST>(y0 - 1 + h.r, x0 - kVEC + h.v * kVEC, nx, ny,
                                                pitch, px, py,
                                                (h.r - t.r) * RM::ROWB + (h.v - t.v) * kVEC * EB);
                    }
            }
        }

        // level-0 planes z0-T .. z1+T-1 are copied; the next one to slot_ld
        PlaneFeed feed(z0 - T, nz, pz);
        const int slot_end = own0 + RING * SLOTB;
        int slot_ld = own0;
        auto issue = [&]() {
            if (feed.n < z1 + T) {
                const ST* g = gin + (long long)feed.plane() * plane;
                unsigned char* const d = smem + slot_ld;
#pragma unroll
                for (int k = 0; k < NF; ++k) {
                    if (k == 0 || !inner_warp)   // (no break: f stays in registers)
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        const ST* gs = vec_at(g, f[k].goff) + s * fstride;
                        const int ok = f[k].mode == 1 &&
                                       RD_DBG_GLOBAL(sd, gs, 4 * (int)sizeof(ST), kSiteCopySrc);
                        Store<ST>::cp_async_if(
                            reinterpret_cast<ST*>(d + f[k].soff + s * RM::SPB), gs, ok);
                    }
                }
                if (elems)   // periodic x, nx not a multiple of 4
#pragma unroll
                    for (int k = 0; k < NF; ++k)
                        fetch_elems<ST, S>(f[k], d, RM::SPB, g, fstride, nx, sd);
            }
            feed.next();
            slot_ld += SLOTB;
            if (slot_ld == slot_end) slot_ld = own0;
            cp_async_commit();
        };
#pragma unroll 1
        for (int j = 0; j < P; ++j) issue();

        // kWindX: the Courant number of the plane being advanced and of the
        // next, loaded a plane ahead
        float cxq = 0.0f, cxn = 0.0f;
        if constexpr (VAR == kWindX) cxn = courant_at(sd, sd.courant, z0);
        // one step of the position's cells in plane q (mapped index zw):
        // centres cen, z neighbours zm / zp, x and y neighbours around ``p``
        auto advance = [&](const float(&zm)[S][kVEC], const float(&cen)[S][kVEC],
                           const float(&zp)[S][kVEC], const unsigned char* p, int q, int zw,
                           float(&o)[S][kVEC]) {
            float inc[S][kVEC];
            react4<M>(sd, cen, inc);
            const float cx = PLAIN || VAR == kWindX ? 0.0f : courant_at(sd, sd.courant, zw);
            const bool src_here = src_col && zw == sd.src_z;
            const unsigned faces = xyf | z_faces(q, nz);
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const unsigned char* ps = p + s * RM::SPB;
                float xm[kVEC], xp[kVEC], ym[kVEC], yp[kVEC];
                lds_vec<ST>(ps - RM::ROWB, ym);
                lds_vec<ST>(ps + RM::ROWB, yp);
                sides.get<ST>(cen[s], ps, xm, xp);
                if constexpr (PLAIN) {
                    euler4_iso(cen[s], xm, xp, ym, yp, zm[s], zp[s], sd.kx[s], inc[s], o[s]);
                } else if constexpr (VAR == kWindX) {
                    // behind the loads, on a copy of its own: a branch ahead of
                    // them holds them up, and the species' writes merged into
                    // one would be indexed in local memory
                    float in[kVEC];
#pragma unroll
                    for (int i = 0; i < kVEC; ++i) in[i] = inc[s][i];
                    if (src_here && s == sd.src_s) {
#pragma unroll
                        for (int i = 0; i < kVEC; ++i)
                            if ((px ? wrapi(xs + i, nx) : xs + i) == sd.src_x)
                                in[i] = __fadd_rn(in[i], sd.src_amt);
                    }
                    if (cxq != 0.0f) {
#pragma unroll
                        for (int i = 0; i < kVEC; ++i)
                            in[i] = __fmaf_rn(-cxq, __fsub_rn(cen[s][i], xm[i]), in[i]);
                    }
                    euler4_aniso(cen[s], xm, xp, ym, yp, zm[s], zp[s], sd.kx[s], sd.ky[s],
                                 sd.kz[s], in, o[s]);
                } else {
                    species_core(sd, s, cen[s], xm, xp, ym, yp, zm[s], zp[s], inc[s], cx, src_here,
                                 px, xs, o[s], cy, cz);
                    held_layers_at(sd, s, faces, xs, y, q, o[s]);
                }
            }
        };

        ST* gst = gout + (long long)z0 * plane + (long long)y * pitch + xs;
        auto store = [&](const float(&o)[S][kVEC]) {
#pragma unroll
            for (int s = 0; s < S; ++s)
                if (stores &&
                    RD_DBG_GLOBAL(sd, gst + s * fstride, 4 * (int)sizeof(ST), kSiteStateStore))
                    Store<ST>::store(gst + s * fstride, o[s]);
            gst += plane;
        };
        // own vectors of three successive planes at both levels, in three
        // sets whose roles rotate from plane to plane
        float A0[S][kVEC], B0[S][kVEC], C0[S][kVEC];
        float A1[S][kVEC], B1[S][kVEC], C1[S][kVEC];
        int slot = own0;                              // ring slot of plane e - 1
        int par1 = 0;                                 // level-1 slot of plane e - 1
        auto next_slot = [&](int x) {
            x += SLOTB;
            return x == slot_end ? own0 : x;
        };
        const int first = z0 - T + 1;
        // the step that advances level 0 of plane e: its planes e - 1, e,
        // e + 1 in m0, c0, p0; T = 2: level 1 of planes e - 2, e - 1, e in
        // m1, c1, p1
        auto body = [&](int e, float(&m0)[S][kVEC], float(&c0)[S][kVEC], float(&p0)[S][kVEC],
                        float(&m1)[S][kVEC], float(&c1)[S][kVEC], float(&p1)[S][kVEC]) {
            // planes through e + 1 must have landed: of those issued, through
            // e + P - 2, all but the newest P - 3
            cp_async_wait<P - 3>();
            __syncthreads();
            const int s1 = next_slot(slot);
            if (T == 2 || inner_warp) {
                const int s2 = next_slot(s1);
                if (e == first) {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        lds_vec<ST>(smem + slot + s * RM::SPB, m0[s]);
                        lds_vec<ST>(smem + s1 + s * RM::SPB, c0[s]);
                    }
                    sides.set_ghost(c0);
                }
#pragma unroll
                for (int s = 0; s < S; ++s) lds_vec<ST>(smem + s2 + s * RM::SPB, p0[s]);
                sides.set_ghost(p0);
            }
            issue();   // after the reads of plane e - 1, whose slot it refills
            if constexpr (T == 1) {
                if constexpr (VAR == kWindX) {
                    cxq = cxn;
                    cxn = courant_at(sd, sd.courant, min(e + 1, nz - 1));
                }
                if (inner_warp) {
                    float o[S][kVEC];
                    advance(m0, c0, p0, smem + s1, e, e, o);
                    store(o);
                }
            } else {
                const int zw = pz ? wrapi(e, nz) : mirror_index(e, nz);
                advance(m0, c0, p0, smem + s1, e, zw, p1);
                unsigned char* const W = smem + own1 + (par1 ^ SLOTB1);
#pragma unroll
                for (int s = 0; s < S; ++s) {
#pragma unroll
                    for (int i = 0; i < kVEC; ++i) p1[s][i] = Store<ST>::round(p1[s][i]);
                    Store<ST>::store(reinterpret_cast<ST*>(W + s * RM::SPB), p1[s]);
                }
                sides.set_ghost(p1);
                if (e > z0 && inner_warp) {
                    float o[S][kVEC];
                    advance(m1, c1, p1, smem + own1 + par1, e - 1, e - 1, o);
                    store(o);
                }
                par1 ^= SLOTB1;
            }
            slot = s1;
        };
        for (int e = first;;) {
            body(e, A0, B0, C0, A1, B1, C1);
            if (++e == z1 + T - 1) break;
            body(e, B0, C0, A0, B1, C1, A1);
            if (++e == z1 + T - 1) break;
            body(e, C0, A0, B0, C1, A1, B1);
            if (++e == z1 + T - 1) break;
        }
        if (ONE && item + gridDim.x >= a.nitems) chain_release();   // the last item
        cp_async_wait<0>();
        __syncthreads();
    }
}

}  // namespace rdk
