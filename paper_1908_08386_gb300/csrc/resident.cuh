// Many coupled steps in one launch with the state kept on the chip.
//
// A grid whose tiles all fit on the SMs at once (one block per SM, one tile
// per block) needs no global memory between steps: each block keeps its tile's
// populations, temperature and velocities in shared memory and exchanges only
// the tile's border with its neighbours, so a step costs the tile's arithmetic
// and one exchange through the L2 instead of a launch, a pipeline fill and a
// drain, which bound small cavities whatever their size.  Measured (us per
// step, one launch per step -> resident, 64 or more steps): FP32 64^2 3.55 -> 1.70,
// 128^2 3.86 -> 1.74, 256^2 4.52 -> 2.23, 384^2 4.81 -> 3.18, 512^2 5.7 -> 5.6; FP16
// 256^2 4.40 -> 2.15; double-single 64^2 5.80 -> 3.46, 128^2 5.82 -> 3.07, 192^2 5.96
// -> 3.62, 256^2 8.5 -> 6.1; FP64 64^2 17.2 -> 5.1, 128^2 17.3 -> 9.2, 192^2 17.4 ->
// 15.7; 512 x 384 with two sub-steps (four launches) 22 -> 8.1, with QUICK and three
// 32 -> 13.
// What bounds it now: the exchange (about 1.1 us) and, for the 64-bit types,
// the dependent chain of one node's operations.
//
// The blocks of a launch wait on one another, so it is a cooperative launch
// (all blocks resident), and every wait is bounded like the other kernels'.
//
// Exchange.  A block posts the border values its neighbours will pull to its
// mailbox in global memory, each as one 64-bit word {32-bit value, 32-bit tag}
// (two words for 64-bit types): a 64-bit access is single-copy atomic, so a
// reader that sees the tag of the step it wants has the value, without fences
// or flags and in one L2 round trip.  Tags count the exchanges of the handle
// since its tile list was built (which clears the mailboxes), and exchanges
// alternate between two slots: a block posts exchange t + 2 into the slot of
// exchange t only after it has read every neighbour's exchange t + 1, which a
// neighbour posts after it has read exchange t.
//
// What is exchanged: population q at a node x is pulled into x + e_q, and a
// block takes the moments of its tile and of the one-node ring around it
// (corners included: an obstacle node's partner may lie there), so it needs
// (q, x) for every x outside the tile with x + e_q in the tile or the ring:
// 2 (TW + 2) + 2 TH values per direction, in bands of 1 + c_q and 1 - c_q rows
// and columns on opposite sides.  Temperature: the ring (and the second row
// and column out for QUICK's far node).
//
// The arithmetic per node is that of the one-launch-per-step kernels, in the
// same order with the same roundings: results are equal bit for bit.
#pragma once

#include "kernels.cuh"

namespace lbmfvm_dev {

template <class S, int TW_, int TH_, int NT_, int RT_>
struct ResTile {
    using C = typename Compute<S>::type;
    static constexpr int TW = TW_, TH = TH_, NT = NT_, RT = RT_;
    static constexpr int BLOCK = NT + RT;        // tile threads, then ring threads
    // Four threads per node (small FP64 tiles, see quad_moments): one direction
    // pair and one face each.
    static constexpr bool QUAD = NT == 4 * TW * TH;
    static constexpr int NPT = QUAD ? 1 : TW * TH / NT;  // own nodes per tile thread
    static constexpr int FW = TW + 4, FH = TH + 4, PL = FW * FH;  // staged box: two nodes around the tile
    static constexpr int RW = TW + 2, RH = TH + 2;
    static constexpr int NRING = 2 * TW + 2 * TH;                 // ring nodes a face can touch (no corners)
    static constexpr int NRT = (NRING + RT - 1) / RT;
    static constexpr bool WIDE = sizeof(S) == 8;                  // two words per value
    // posted values: per direction the tile's border as its neighbours pull it,
    // then the temperature border and (QUICK) the second temperature border
    static constexpr int SQ = 2 * TW + 2 * (TH - 2), ST2 = 2 * TW + 2 * TH;
    static constexpr int SF = 9 * SQ, ST = SQ + ST2;
    static constexpr int PACKETS = SF + ST;
    static constexpr size_t MAIL_BYTES = 2 * (size_t)PACKETS * (WIDE ? 16 : 8);  // two slots
    // read values
    static constexpr int RQ = 2 * (TW + 2) + 2 * TH, RT2 = 2 * TW + 2 * TH;
    static constexpr int RF = 9 * RQ, RTT = RQ + RT2;
    // posts and reads per thread
    static constexpr int NSF = (SF + BLOCK - 1) / BLOCK, NRF = (RF + BLOCK - 1) / BLOCK;
    static constexpr int NST = (ST + BLOCK - 1) / BLOCK, NRD = (RTT + BLOCK - 1) / BLOCK;
    static constexpr size_t a16(size_t v) { return (v + 15) & ~(size_t)15; }
    static constexpr size_t F_OFF = 0, T_OFF = a16(9 * (size_t)PL * sizeof(S));
    static constexpr size_t U_OFF = T_OFF + a16(2 * (size_t)PL * sizeof(C));
    static constexpr size_t W_OFF = U_OFF + a16(2 * (size_t)RW * RH * sizeof(C));
    static constexpr size_t SMEM = W_OFF + a16(10 * sizeof(C));
    static_assert((QUAD || (TW * TH % NT == 0 && NT % TW == 0)) && NT % 32 == 0 && RT % 32 == 0 && BLOCK <= 1024, "threads");
    static_assert(SMEM <= 230000, "shared memory");
};

// Border maps.  send_node: the node that posted value i of direction (dx, dy)
// holds; read_node: the node (outside the tile) that read value i of direction
// (dx, dy) holds; post_index: the posted index of a tile's node (x, y), which
// must be one a neighbour reads.  Direction (0, 0) is also the temperature's.
template <int TW, int TH>
__host__ __device__ inline void send_node(int i, int dx, int dy, int &x, int &y) {
    if (i < 2 * TW) {
        const int k = i / TW;
        x = i - k * TW;
        y = k < 1 - dy ? k : TH - 2 + k;
    } else {
        const int j = i - 2 * TW, k = j & 1;
        y = 1 - dy + (j >> 1);
        x = k < 1 - dx ? k : TW - 2 + k;
    }
}
template <int TW, int TH>
__host__ __device__ inline void read_node(int i, int dx, int dy, int &x, int &y) {
    if (i < 2 * (TW + 2)) {
        const int k = i / (TW + 2);
        x = i - k * (TW + 2) - 1 - dx;
        y = k < 1 + dy ? k - (1 + dy) : TH + k - (1 + dy);
    } else {
        const int j = i - 2 * (TW + 2), k = j & 1;
        y = j >> 1;
        x = k < 1 + dx ? k - (1 + dx) : TW + k - (1 + dx);
    }
}
template <int TW, int TH>
__host__ __device__ inline int post_index(int x, int y, int dx, int dy) {
    if (y < 1 - dy) return y * TW + x;
    if (y >= TH - 1 - dy) return (y - TH + 2) * TW + x;
    return 2 * TW + 2 * (y - (1 - dy)) + (x < 1 - dx ? x : x - TW + 2);
}
// Second temperature border: rows 1 and TH - 2, columns 1 and TW - 2; read
// from rows -2 and TH + 1, columns -2 and TW + 1.
template <int TW, int TH>
__host__ __device__ inline void send_node2(int i, int &x, int &y) {
    if (i < 2 * TW) {
        const int k = i / TW;
        x = i - k * TW;
        y = k ? TH - 2 : 1;
    } else {
        const int j = i - 2 * TW;
        y = j >> 1;
        x = (j & 1) ? TW - 2 : 1;
    }
}
template <int TW, int TH>
__host__ __device__ inline void read_node2(int i, int &x, int &y) {
    if (i < 2 * TW) {
        const int k = i / TW;
        x = i - k * TW;
        y = k ? TH + 1 : -2;
    } else {
        const int j = i - 2 * TW;
        y = j >> 1;
        x = (j & 1) ? TW + 1 : -2;
    }
}
template <int TW, int TH>
__host__ __device__ inline int post_index2(int x, int y, bool row) {
    if (row) return (y == 1 ? 0 : TW) + x;
    return 2 * TW + 2 * y + (x == 1 ? 0 : 1);
}

namespace mail {

__device__ __forceinline__ uint32_t bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t bits(__half v) { return __half_as_ushort(v); }
__device__ __forceinline__ uint32_t bits(__nv_bfloat16 v) { return __bfloat16_as_ushort(v); }
__device__ __forceinline__ uint2 bits2(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return make_uint2((uint32_t)b, (uint32_t)(b >> 32));
}
__device__ __forceinline__ uint2 bits2(dsf v) { return make_uint2(__float_as_uint(v.hi), __float_as_uint(v.lo)); }
__device__ __forceinline__ void put(float *p, uint32_t b, uint32_t) { *p = __uint_as_float(b); }
__device__ __forceinline__ void put(__half *p, uint32_t b, uint32_t) { *p = __ushort_as_half((unsigned short)b); }
__device__ __forceinline__ void put(__nv_bfloat16 *p, uint32_t b, uint32_t) {
    *p = __ushort_as_bfloat16((unsigned short)b);
}
__device__ __forceinline__ void put(double *p, uint32_t lo, uint32_t hi) {
    *p = __longlong_as_double((long long)(((unsigned long long)hi << 32) | lo));
}
__device__ __forceinline__ void put(dsf *p, uint32_t hi, uint32_t lo) {
    *p = dsf(__uint_as_float(hi), __uint_as_float(lo));
}

__device__ __forceinline__ uint64_t word(uint32_t v, uint32_t tag) { return ((uint64_t)tag << 32) | v; }

// Post value v as packet e of a slot.
template <class V>
__device__ __forceinline__ void post(uint64_t *slot, int e, V v, uint32_t tag) {
    if constexpr (sizeof(V) == 8) {
        const uint2 b = bits2(v);
        asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(slot + 2 * e), "l"(word(b.x, tag)),
                     "l"(word(b.y, tag))
                     : "memory");
    } else {
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(slot + e), "l"(word(bits(v), tag)) : "memory");
    }
}
template <bool WIDE>
struct Packet {
    uint64_t a, b;
    __device__ __forceinline__ void load(const uint64_t *slot, int e) {
        if constexpr (WIDE)
            asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(slot + 2 * e) : "memory");
        else
            asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(a) : "l"(slot + e) : "memory");
    }
    __device__ __forceinline__ bool is(uint32_t tag) const {
        return (uint32_t)(a >> 32) == tag && (!WIDE || (uint32_t)(b >> 32) == tag);
    }
    template <class V>
    __device__ __forceinline__ void to(V *p) const {
        put(p, (uint32_t)a, WIDE ? (uint32_t)b : 0u);
    }
};

}  // namespace mail

// A node's arithmetic split over four neighbouring lanes, s = 0..3.  An FP64
// instruction holds its quarter of an SM for some 80 cycles whatever it
// computes, and a 32-node tile is one warp: one quarter works, the others wait.
// With a lane per direction pair and per face a warp executes about 70 of them
// a step instead of 170, on all four quarters.  Same operations in the same
// order, so the same bits.  64^2 FP64: 8.6 -> 5.0 us per step.  Larger tiles
// fill the quarters as they are.
template <class C>
__device__ __forceinline__ C quad_pick(int s, C a, C b, C c, C d) {
    return s < 2 ? (s == 0 ? a : b) : (s == 2 ? c : d);
}
template <class C>
__device__ __forceinline__ C quad_get(C v, int s) {
    return __shfl_sync(0xffffffffu, v, s, 4);
}
template <class C>
__device__ __forceinline__ void quad_moments(const C g[9], int s, C &drho, C &ux, C &uy) {
    const C p = quad_pick(s, g[0], g[2], g[4], g[6]) + quad_pick(s, g[1], g[3], g[5], g[7]);
    const C q = (quad_pick(s, g[1], g[3], g[2], g[4]) + quad_pick(s, g[5], g[6], g[5], g[7])) +
                quad_pick(s, g[8], g[7], g[6], g[8]);
    drho = ((quad_get(p, 0) + quad_get(p, 1)) + (quad_get(p, 2) + quad_get(p, 3))) + g[8];
    const C jx = quad_get(q, 0) - quad_get(q, 1), jy = quad_get(q, 2) - quad_get(q, 3);
    const C inv = recip(C(1) + drho);
    ux = mul_r(jx, inv);
    uy = mul_r(jy, inv);
}
// nee for the lane's pair (f, b) and the rest population.
template <class C>
__device__ __forceinline__ void quad_nee(C &g0, C &f, C &b, int s, C drho, C &ux, C &uy, C uw, C vw) {
    const C rho = C(1) + drho;
    const C dP0 = mul_r(C(-1.5f), fma_c(uw, uw, mul_r(vw, vw)) - fma_c(ux, ux, mul_r(uy, uy)));
    if (s == 0) g0 = fma_c(mul_r(rho, wq<C>(0)), dP0, g0);
    const C euw = quad_pick(s, uw, vw, uw + vw, vw - uw), euf = quad_pick(s, ux, uy, ux + uy, uy - ux);
    const C A = fma_c(C(4.5f), fma_c(euw, euw, -mul_r(euf, euf)), dP0), B = triple(euw - euf);
    const C rw = mul_r(rho, s < 2 ? wq<C>(1) : wq<C>(5));
    f = fma_c(rw, A + B, f);
    b = fma_c(rw, A - B, b);
    ux = uw;
    uy = vw;
}
// collide for the lane's pair, store(q, value); the rest population by lane 0.
template <class C, class Store>
__device__ __forceinline__ void quad_collide(C g0, C f, C b, int s, C drho, C ux, C uy, C omega, C Gx, C Gy,
                                             Store store) {
    const C rho = C(1) + drho;
    const C P0 = mul_r(C(-1.5f), fma_c(ux, ux, mul_r(uy, uy)));
    const C c = mul_r(C(3), rho);
    const C sx = mul_r(c, Gx), sy = mul_r(c, Gy);
    const C nGu = -fma_c(sx, ux, mul_r(sy, uy));
    const C om1 = C(1) - omega;
    auto out = [&](int q, C w, C gq, C P, C z) {
        store(q, fma_c(om1, gq, mul_r(w, fma_c(P, fma_c(omega, rho, z), fma_c(omega, drho, z)))));
    };
    const C eu = quad_pick(s, ux, uy, ux + uy, uy - ux), es = quad_pick(s, sx, sy, sx + sy, sy - sx);
    const C A = fma_c(C(4.5f), mul_r(eu, eu), P0), B = triple(eu), w = s < 2 ? wq<C>(1) : wq<C>(5);
    out(s < 2 ? 1 + s : 3 + s, w, f, A + B, nGu + es);
    out(s < 2 ? 3 + s : 5 + s, w, b, A - B, nGu - es);
    if (s == 0) out(0, wq<C>(0), g0, P0, nGu);
}

// Limit of the waits in which a block may still be kept off its SM by other work.
constexpr uint64_t kStartWaitNs = 120 * kWaitLimitNs;

// Arguments of a resident launch: steps from the state a.fin, a.Tin to a.fout,
// a.Tout (other buffers), on one tile per block.
template <class S>
struct ResArgs {
    StepArgs<S> a;
    const uint8_t *fflags;
    const CavityDesc *cavs;
    const TileHeader *tiles;  // blockIdx-th: this block's tile; a cavity's tiles row by row
    uint64_t *mailbox;
    uint32_t seq0;            // exchanges before this launch
    int nsteps;
    int quick;                // QUICK face values (general form)
    int tile_w, tile_h;       // tiles of the step kernel
    int *ctr[2];              // tile counters of the step kernel's lists, cleared for the next launch
    uint32_t spoil;           // test hook: block 0's border values carry tags that nobody waits for
    uint64_t late_ns;         // test hook: block 0 starts this much later
    // limits of a wait: while a block may still be kept off its SM by other work,
    // and once every block runs
    uint64_t start_ns, wait_ns;
};

// GENERAL: QUICK face values and energy sub-steps; else the central update,
// one per step.  BORDERS: a tile may hold a row border of the step kernel's tiles
// beside a wall (bits 23 and 24 of info below).  FP32 arithmetic in tiles of more
// than 8 rows (64-bit types round the two wall velocities alike; the step
// kernel's tiles have 8 rows or more).  Us per step without / with it: 256^2 in
// 32 x 16 2.21 / 2.23, 384^2 in 32 x 32 3.15 / 3.15, 512^2 in 64 x 32 5.55 / 5.8,
// 512 x 384 with two sub-steps 8.07 / 8.5: a form of its own in the last shapes.
template <class S, class G>
constexpr bool res_borders() {
    return std::is_same<typename Compute<S>::type, float>::value && G::TH > 8;
}
template <class S, class G>
constexpr bool res_borders_apart() {
    return res_borders<S, G>() && G::NPT > 2;
}
struct ResForm {
    bool general, borders;
};
template <class S, class G, bool GENERAL, bool BORDERS>
__global__ void __launch_bounds__(G::BLOCK, 1) resident_kernel(const ResArgs<S> r) {
    using C = typename Compute<S>::type;
    constexpr int TW = G::TW, TH = G::TH, FW = G::FW, PL = G::PL, RW = G::RW, NPT = G::NPT, BLOCK = G::BLOCK;
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ int gave_up;
    S *F = reinterpret_cast<S *>(rsm + G::F_OFF);
    C *T = reinterpret_cast<C *>(rsm + G::T_OFF);  // two planes
    C *RU = reinterpret_cast<C *>(rsm + G::U_OFF), *RV = RU + RW * G::RH;
    C *wall = reinterpret_cast<C *>(rsm + G::W_OFF);  // velocity of sides W, E, S, N and of obstacles (rest)
    const int tid = threadIdx.x;
    const TileHeader &hd = r.tiles[blockIdx.x];
    const int x0 = hd.x0, y0 = hd.y0, ox = hd.ox, oy = hd.oy, cnx = hd.nx, cny = hd.ny;
    const int m = GENERAL ? hd.substeps : 1;
    C alpha, omega, gbeta, t_ref, fx, fy, dt;
    if constexpr (std::is_same<C, double>::value) {
        alpha = hd.alpha, omega = hd.omega, gbeta = hd.gbeta, t_ref = hd.t_ref, fx = hd.fx, fy = hd.fy;
    } else if constexpr (std::is_same<C, dsf>::value) {
        alpha = dsf(hd.alpha_f, hd.alpha_lo), omega = dsf(hd.omega_f, hd.omega_lo);
        gbeta = dsf(hd.gbeta_f, hd.gbeta_lo), t_ref = dsf(hd.t_ref_f, hd.t_ref_lo);
        fx = dsf(hd.fx_f, hd.fx_lo), fy = dsf(hd.fy_f, hd.fy_lo);
    } else {
        alpha = hd.alpha_f, omega = hd.omega_f, gbeta = hd.gbeta_f, t_ref = hd.t_ref_f, fx = hd.fx_f, fy = hd.fy_f;
    }
    dt = TileParams<C>::dt(hd);
    const CavityDesc &cv = r.cavs[hd.cav];
    const int pitch = r.a.pitch;
    const long long plane = r.a.plane;
    const long long org = (long long)y0 * pitch + x0;  // the tile's first node
    auto in_cavity = [&](int lx, int ly) {
        return ox + lx >= 0 && ox + lx < cnx && oy + ly >= 0 && oy + ly < cny;
    };
    auto fi = [&](int lx, int ly) { return (ly + 2) * FW + lx + 2; };
    auto side_of = [&](int lx, int ly, uint8_t c) {
        if ((c >> 6) == TH_OBSTACLE) return 4;
        const int x = ox + lx, y = oy + ly;
        return x == 0 ? 0 : (x == cnx - 1 ? 1 : (y == 0 ? 2 : 3));
    };

    if (r.late_ns && blockIdx.x == 0)
        for (const uint64_t t0 = tma::globaltimer(); tma::globaltimer() - t0 < r.late_ns;) __nanosleep(1000);

    // The staged box of the state to start from (nothing outside the cavity).
    for (int i = tid; i < PL; i += BLOCK) {
        const int lx = i % FW - 2, ly = i / FW - 2;
        const bool in = in_cavity(lx, ly);
        const long long k = org + (long long)ly * pitch + lx;
#pragma unroll
        for (int q = 0; q < 9; q++) {
            if (in) F[q * PL + i] = r.a.fin[k + q * plane];
            else st(F + q * PL + i, C(0));
        }
        T[i] = T[PL + i] = in ? r.a.Tin[k] : C(0);
    }
    for (int i = tid; i < RW * G::RH; i += BLOCK) RU[i] = RV[i] = C(0);
    if (tid < 5) {
        if constexpr (std::is_same<C, float>::value) {
            wall[2 * tid] = tid < 4 ? cv.wall_uf[tid] : 0.0f;
            wall[2 * tid + 1] = tid < 4 ? cv.wall_vf[tid] : 0.0f;
        } else {
            wall[2 * tid] = tid < 4 ? C(cv.wall_u[tid]) : C(0);
            wall[2 * tid + 1] = tid < 4 ? C(cv.wall_v[tid]) : C(0);
        }
    }
    if (tid == 0) {
        gave_up = 0;
        if (blockIdx.x == 0)
            for (int l = 0; l < 2; l++) r.ctr[l][0] = r.ctr[l][1] = 0;
    }

    // own node j of this thread, and its lane of the four that share it
    auto own_node = [&](int j) { return G::QUAD ? tid >> 2 : tid + j * G::NT; };
    const int lane4 = tid & 3;

    // Own nodes: code, face flags, far-face flags (QUICK), wall side; bits 23 and
    // 24: the node above (below) is a wall node across a border of the step
    // kernel's tiles inside this one, see the ring nodes below.  (The step kernel's
    // borders between columns are borders of these tiles too, and the two nodes
    // of a face between wall nodes lie on one side.)
    const bool computes = tid < G::NT;
    uint32_t info[NPT];
    constexpr uint32_t kDead = CODE_OUTSIDE;
#pragma unroll
    for (int j = 0; j < NPT; j++) {
        info[j] = kDead;
        const int i = own_node(j), ly = i / TW, lx = i - ly * TW;
        if (computes && in_cavity(lx, ly)) {
            const long long k = org + (long long)ly * pitch + lx;
            const uint8_t c = decode(r.a.code[k]);
            const uint8_t ff = r.fflags[k];
            uint32_t far = 0;
            if (GENERAL) {
                if ((ff & FF_OPEN_E) && (r.fflags[k + 1] & FF_OPEN_E)) far |= FF_OPEN_E;
                if ((ff & FF_OPEN_W) && (r.fflags[k - 1] & FF_OPEN_W)) far |= FF_OPEN_W;
                if ((ff & FF_OPEN_N) && (r.fflags[k + pitch] & FF_OPEN_N)) far |= FF_OPEN_N;
                if ((ff & FF_OPEN_S) && (r.fflags[k - pitch] & FF_OPEN_S)) far |= FF_OPEN_S;
            }
            info[j] = c | ((uint32_t)ff << 8) | (far << 16) | ((uint32_t)side_of(lx, ly, c) << 20);
            if (BORDERS && m == 1) {
                const int y = oy + ly;
                if (ly + 1 < TH && (ff & FF_OPEN_N) && (y + 1) % r.tile_h == 0 && (decode(r.a.code[k + pitch]) & 3) == KIND_WALL)
                    info[j] |= 1u << 23;
                if (ly > 0 && (ff & FF_OPEN_S) && y % r.tile_h == 0 && (decode(r.a.code[k - pitch]) & 3) == KIND_WALL)
                    info[j] |= 1u << 24;
            }
            if ((c & 3) == KIND_SOLID) {
                // inert nodes never change: their results are written once
#pragma unroll
                for (int q = 0; q < 9; q++) st(r.a.fout + k + q * plane, C(0));
                r.a.Tout[k] = r.a.Tin[k];
            }
        }
    }
    // Ring nodes of the ring threads.  Fluid ones are pulled every step.  The
    // step kernel takes a wall node's velocity from its extrapolated
    // populations inside a tile of its own and from the wall across a border
    // of its tiles (the two differ by rounding); so does this one, at the step
    // kernel's borders, so that both round alike.
    auto ring_node = [&](int i, int &lx, int &ly) {
        if (i < TW) lx = i, ly = -1;
        else if (i < 2 * TW) lx = i - TW, ly = TH;
        else lx = ((i - 2 * TW) & 1) ? TW : -1, ly = (i - 2 * TW) >> 1;
    };
    uint32_t ring_fluid = 0, ring_wall = 0, rinfo[G::NRT];
    __syncthreads();  // RU, RV cleared, walls set
    if (!computes) {
#pragma unroll
        for (int j = 0; j < G::NRT; j++) {
            const int i = tid - G::NT + j * G::RT;
            int lx, ly;
            ring_node(i, lx, ly);
            rinfo[j] = 0;
            if (i >= G::NRING || !in_cavity(lx, ly)) continue;
            const uint8_t c = decode(r.a.code[org + (long long)ly * pitch + lx]);
            if ((c & 3) == KIND_FLUID) ring_fluid |= 1u << j;
            if ((c & 3) == KIND_WALL) {
                const int sd = side_of(lx, ly, c), d = partner_dir(c);
                const int px = lx + cx_rt(d), py = ly + cy_rt(d);
                // (the sub-step path's velocity planes hold the extrapolated ones throughout)
                const bool border = m == 1 && (lx < 0     ? ox % r.tile_w == 0
                                               : lx >= TW ? (ox + TW) % r.tile_w == 0
                                               : ly < 0   ? oy % r.tile_h == 0
                                                          : (oy + TH) % r.tile_h == 0);
                // (an obstacle surface has no open face; its partner may lie too far out to be pulled)
                if (!border && sd < 4 && px >= -1 && px <= TW && py >= -1 && py <= TH) ring_wall |= 1u << j;
                rinfo[j] = c | ((uint32_t)sd << 20);
                RU[(ly + 1) * RW + lx + 1] = wall[2 * sd];
                RV[(ly + 1) * RW + lx + 1] = wall[2 * sd + 1];
            }
        }
    }

    // Where this thread's posts come from and its reads go to.  A read takes
    // a packet index of the neighbour's mailbox (-1: nothing there).
    constexpr int NSF = G::NSF, NRF = G::NRF, NST = G::NST, NRD = G::NRD;
    int sf[NSF], rf_at[NRF], rf_to[NRF], rt_at[NRD], rt_to[NRD];
    const int ntx = (cnx + TW - 1) / TW, nty = (cny + TH - 1) / TH;
    const int reach = ntx > nty ? ntx : nty;  // steps by which every block of the cavity has been waited for
    auto packet_of = [&](int lx, int ly, auto index) {  // of node (lx, ly) outside the tile
        if (!in_cavity(lx, ly)) return -1;
        const int dx = lx < 0 ? -1 : (lx >= TW ? 1 : 0), dy = ly < 0 ? -1 : (ly >= TH ? 1 : 0);
        const int t = (int)blockIdx.x + dx + dy * ntx;
        return t * 2 * G::PACKETS + index(lx - dx * TW, ly - dy * TH);
    };
#pragma unroll
    for (int i = 0; i < NSF; i++) {
        const int e = tid + i * BLOCK, q = e / G::SQ;
        int x = 0, y = 0;
        if (e < G::SF) send_node<TW, TH>(e - q * G::SQ, cx_rt(q), cy_rt(q), x, y);
        sf[i] = e < G::SF ? q * PL + fi(x, y) : -1;
    }
#pragma unroll
    for (int i = 0; i < NRF; i++) {
        const int e = tid + i * BLOCK, q = e / G::RQ;
        rf_at[i] = -1;
        rf_to[i] = 0;
        if (e < G::RF) {
            const int dx = cx_rt(q), dy = cy_rt(q);
            int x, y;
            read_node<TW, TH>(e - q * G::RQ, dx, dy, x, y);
            rf_at[i] = packet_of(x, y, [&](int a, int b) { return q * G::SQ + post_index<TW, TH>(a, b, dx, dy); });
            rf_to[i] = q * PL + fi(x, y);
        }
    }
#pragma unroll
    for (int i = 0; i < NRD; i++) {
        const int e = tid + i * BLOCK;
        rt_at[i] = -1;
        rt_to[i] = 0;
        int x, y;
        if (e < G::RQ) {
            read_node<TW, TH>(e, 0, 0, x, y);
            rt_at[i] = packet_of(x, y, [&](int a, int b) { return G::SF + post_index<TW, TH>(a, b, 0, 0); });
            rt_to[i] = fi(x, y);
        } else if (GENERAL && r.quick && e < G::RTT) {
            read_node2<TW, TH>(e - G::RQ, x, y);
            const bool row = e - G::RQ < 2 * TW;
            rt_at[i] = packet_of(x, y, [&](int a, int b) { return G::SF + G::SQ + post_index2<TW, TH>(a, b, row); });
            rt_to[i] = fi(x, y);
        }
    }
    constexpr int WORDS = G::WIDE ? 2 : 1;
    uint64_t *own = r.mailbox + (size_t)blockIdx.x * 2 * G::PACKETS * WORDS;
    auto post_T = [&](const C *Tn, uint32_t tag) {
        uint64_t *slot = own + (size_t)(tag & 1u) * G::PACKETS * WORDS;
#pragma unroll
        for (int i = 0; i < NST; i++) {
            const int e = tid + i * BLOCK;
            int x, y;
            if (e < G::SQ) send_node<TW, TH>(e, 0, 0, x, y);
            else if (GENERAL && r.quick && e < G::ST) send_node2<TW, TH>(e - G::SQ, x, y);
            else continue;
            mail::post(slot, G::SF + e, Tn[fi(x, y)], tag);
        }
    };
    // Reads N packets of the slot of `tag` into base + to[i] in step k; false when
    // a wait ran out.
    auto read = [&](auto *base, const int *at, const int *to, auto count, uint32_t tag, int k) {
        constexpr int N = decltype(count)::value;
        const uint64_t *slot = r.mailbox + (size_t)(tag & 1u) * G::PACKETS * WORDS;
        uint64_t t0 = 0;
        uint32_t left = 0;
#pragma unroll
        for (int i = 0; i < N; i++)
            if (at[i] >= 0) left |= 1u << i;
        for (uint32_t it = 0; left; it++) {
            mail::Packet<G::WIDE> p[N];
#pragma unroll
            for (int i = 0; i < N; i++)
                if (left >> i & 1u) p[i].load(slot, at[i]);
#pragma unroll
            for (int i = 0; i < N; i++)
                if ((left >> i & 1u) && p[i].is(tag)) {
                    p[i].to(base + to[i]);
                    left &= ~(1u << i);
                }
            if ((it & 63u) == 63u) {
                const uint64_t t = tma::globaltimer();
                if (t0 == 0) t0 = t;
                // an exchange is between neighbours: a block that starts late
                // holds up those d tiles away in exchange d - 1
                else if (t - t0 > (k < reach ? r.start_ns : r.wait_ns)) return false;
            }
        }
        return true;
    };
    auto pull = [&](int lx, int ly, C g[9]) {
        const S *p = F + fi(lx, ly);
#pragma unroll
        for (int q = 0; q < 9; q++) g[q] = ld(p + q * PL - cy(q) * FW - cx(q));
    };

    const uint32_t spoil = blockIdx.x == 0 ? r.spoil : 0u;

    int cb = 0;  // temperature plane of the current step
    for (int k = 0; k < r.nsteps; k++) {
        // Phase A: moments of the own nodes (kept in registers) and of the ring.
        C g[NPT][9], dr[NPT], uu[NPT], vv[NPT], Tn[NPT];
        C qf, qb;  // the lane's pair of populations (four threads per node)
        if (computes) {
#pragma unroll
            for (int j = 0; j < NPT; j++) {
                const int i = own_node(j), ly = i / TW, lx = i - ly * TW;
                const uint32_t c = info[j];
                const int kind = c & 3;
                if constexpr (G::QUAD) {
                    const int d = kind == KIND_WALL ? partner_dir((uint8_t)c) : 0;
                    pull(lx + cx_rt(d), ly + cy_rt(d), g[j]);  // inert nodes hold zeros
                    quad_moments<C>(g[j], lane4, dr[j], uu[j], vv[j]);
                    qf = quad_pick(lane4, g[j][1], g[j][2], g[j][5], g[j][6]);
                    qb = quad_pick(lane4, g[j][3], g[j][4], g[j][7], g[j][8]);
                    if (kind == KIND_WALL) {
                        const int sd = (c >> 20) & 7;
                        quad_nee<C>(g[j][0], qf, qb, lane4, dr[j], uu[j], vv[j], wall[2 * sd], wall[2 * sd + 1]);
                    }
                    if (kind == KIND_SOLID) uu[j] = vv[j] = C(0);
                } else if (kind != KIND_SOLID) {
                    // a warp of fluid and wall nodes pulls and sums once (a
                    // wall node from its partner)
                    const int d = kind == KIND_WALL ? partner_dir((uint8_t)c) : 0;
                    pull(lx + cx_rt(d), ly + cy_rt(d), g[j]);
                    moments<C>(g[j], dr[j], uu[j], vv[j]);
                    if (kind == KIND_WALL) {
                        const int sd = (c >> 20) & 7;
                        nee<C>(g[j], dr[j], uu[j], vv[j], wall[2 * sd], wall[2 * sd + 1]);
                    }
                } else {
                    uu[j] = vv[j] = C(0);
                }
                RU[(ly + 1) * RW + lx + 1] = uu[j];
                RV[(ly + 1) * RW + lx + 1] = vv[j];
            }
        } else {
#pragma unroll
            for (int j = 0; j < G::NRT; j++) {
                if (!((ring_fluid | ring_wall) >> j & 1u)) continue;
                int lx, ly;
                ring_node(tid - G::NT + j * G::RT, lx, ly);
                C h[9], hd_, hu, hv;
                const bool w = ring_wall >> j & 1u;
                const int d = w ? partner_dir((uint8_t)rinfo[j]) : 0;
                pull(lx + cx_rt(d), ly + cy_rt(d), h);
                moments<C>(h, hd_, hu, hv);
                if (w) {
                    const int sd = rinfo[j] >> 20;
                    nee<C>(h, hd_, hu, hv, wall[2 * sd], wall[2 * sd + 1]);
                }
                RU[(ly + 1) * RW + lx + 1] = hu;
                RV[(ly + 1) * RW + lx + 1] = hv;
            }
        }
        __syncthreads();
        // Phase B: energy balance (in m sub-steps) and collision.
        const bool last = k + 1 == r.nsteps;
        bool ok = true;
        for (int s = 1; s <= m; s++) {
            const C *Tc = T + cb * PL;
            C *To = T + (cb ^ 1) * PL;
            if (computes) {
#pragma unroll
                for (int j = 0; j < NPT; j++) {
                    const uint32_t c = info[j];
                    if (!(G::QUAD && !GENERAL) && (c & 3) == KIND_SOLID) continue;
                    const int i = own_node(j), ly = i / TW, lx = i - ly * TW;
                    const int t = fi(lx, ly), rr = (ly + 1) * RW + lx + 1, th = (c >> 6) & 3;
                    const C TP = Tc[t];
                    C t1 = TP;
                    if constexpr (G::QUAD && !GENERAL) {
                        // lanes E, W, N, S: one face each, summed as fv_update does
                        const bool vert = lane4 >= 2, minus = (lane4 & 1) == 0;
                        const int step = lane4 & 1 ? -1 : 1;
                        const C Tb = Tc[t + step * (vert ? FW : 1)];
                        const C wb = vert ? RV[rr + step * RW] : RU[rr + step], wP = vert ? vv[j] : uu[j];
                        const C pr = mul_r(C(0.25f) * (wP + wb), TP + Tb);
                        const uint32_t ff = c >> 8;
                        const uint32_t bit = vert ? (minus ? FF_OPEN_N : FF_OPEN_S) : (minus ? FF_OPEN_E : FF_OPEN_W);
                        const C f = ff & bit ? fma_c(alpha, Tb - TP, minus ? -pr : pr) : C(0);
                        const C fe = quad_get(f, 0), fw = quad_get(f, 1), fn = quad_get(f, 2), fs = quad_get(f, 3);
                        if (th == TH_FV) {
                            const C ex = ((ff & FF_IN_W) ? C(0.5) : C(0)) + ((ff & FF_IN_E) ? C(0.5) : C(0));
                            const C ey = ((ff & FF_IN_S) ? C(0.5) : C(0)) + ((ff & FF_IN_N) ? C(0.5) : C(0));
                            const C inv_v = (ex < C(1) ? C(2) : C(1)) * (ey < C(1) ? C(2) : C(1));
                            t1 = TP + (ey * (fe + fw) + ex * (fn + fs)) * inv_v;
                        } else if (th == TH_OBSTACLE) {
                            const int d = partner_dir((uint8_t)c);
                            t1 = Tc[t + cy_rt(d) * FW + cx_rt(d)];
                        }
                    } else if (th == TH_FV) {
                        const uint32_t ff = c >> 8, far = c >> 16;
                        const C ex = ((ff & FF_IN_W) ? C(0.5) : C(0)) + ((ff & FF_IN_E) ? C(0.5) : C(0));
                        const C ey = ((ff & FF_IN_S) ? C(0.5) : C(0)) + ((ff & FF_IN_N) ? C(0.5) : C(0));
                        const C TE = Tc[t + 1], TWt = Tc[t - 1], TN = Tc[t + FW], TS = Tc[t - FW];
                        const C uE = RU[rr + 1], uW = RU[rr - 1];
                        C vN, vS;
                        if constexpr (BORDERS && NPT <= 2) {
                            const C *wv = wall + 2 * ((c >> 20) & 7) + 1;
                            vN = *(c >> 23 & 1u ? wv : RV + rr + RW);
                            vS = *(c >> 24 & 1u ? wv : RV + rr - RW);
                        } else {
                            vN = RV[rr + RW];
                            vS = RV[rr - RW];
                            if (BORDERS && (c >> 23 & 3u)) {  // (two addresses more per node would spill)
                                const C wv = wall[2 * ((c >> 20) & 7) + 1];
                                if (c >> 23 & 1u) vN = wv;
                                if (c >> 24 & 1u) vS = wv;
                            }
                        }
                        const bool oE = ff & FF_OPEN_E, oN = ff & FF_OPEN_N, oW = ff & FF_OPEN_W, oS = ff & FF_OPEN_S;
                        if (!GENERAL || (!r.quick && m == 1)) {
                            t1 = fv_update<C>(TP, uu[j], vv[j], ex, ey, alpha, oE, TE, uE, oN, TN, vN, oW, TWt, uW, oS,
                                              TS, vS);
                        } else {
                            C fE, fW, fN, fS;
                            if (r.quick) {
                                fE = quick_face<C>(uu[j] + uE, TP, TE, oW, TWt, far & FF_OPEN_E, Tc[t + 2]);
                                fW = quick_face<C>(-(uu[j] + uW), TP, TWt, oE, TE, far & FF_OPEN_W, Tc[t - 2]);
                                fN = quick_face<C>(vv[j] + vN, TP, TN, oS, TS, far & FF_OPEN_N, Tc[t + 2 * FW]);
                                fS = quick_face<C>(-(vv[j] + vS), TP, TS, oN, TN, far & FF_OPEN_S, Tc[t - 2 * FW]);
                            } else {
                                fE = C(0.5) * (TP + TE);
                                fW = C(0.5) * (TP + TWt);
                                fN = C(0.5) * (TP + TN);
                                fS = C(0.5) * (TP + TS);
                            }
                            t1 = fv_update_faces<C>(TP, uu[j], vv[j], ex, ey, alpha, dt, oE, TE, uE, fE, oN, TN, vN, fN,
                                                    oW, TWt, uW, fW, oS, TS, vS, fS);
                        }
                    } else if (th == TH_OBSTACLE) {
                        const int d = partner_dir((uint8_t)c);
                        t1 = Tc[t + cy_rt(d) * FW + cx_rt(d)];
                    }
                    To[t] = t1;
                    Tn[j] = t1;
                }
            }
            cb ^= 1;
            if (s < m) {
                const uint32_t tag = (r.seq0 + (uint32_t)k) * (uint32_t)m + (uint32_t)s;
                __syncthreads();
                post_T(To, tag ^ spoil);
                ok &= read(To, rt_at, rt_to, std::integral_constant<int, NRD>{}, tag, k);
                if (!ok) gave_up = 1;
                __syncthreads();
                // (the last step makes no other exchange that would report it)
                if (gave_up) {
                    if (!ok) atomicOr(r.a.err, kErrTimeout);
                    return;
                }
            }
        }
        if (computes) {
#pragma unroll
            for (int j = 0; j < NPT; j++) {
                const uint32_t c = info[j];
                if ((c & 3) == KIND_SOLID) continue;
                const int i = own_node(j), ly = i / TW, lx = i - ly * TW;
                const C Gy = fma_c(gbeta, Tn[j] - t_ref, fy);
                if constexpr (G::QUAD) {
                    const long long kk = org + (long long)ly * pitch + lx;
                    S *out = last ? r.a.fout + kk : F + fi(lx, ly);
                    const long long pl = last ? plane : PL;
                    if (last) r.a.Tout[kk] = Tn[j];
                    quad_collide<C>(g[j][0], qf, qb, lane4, dr[j], uu[j], vv[j], omega, fx, Gy,
                                    [&](int q, C v) { st(out + q * pl, v); });
                } else if (last) {
                    const long long kk = org + (long long)ly * pitch + lx;
                    S *out = r.a.fout + kk;
                    r.a.Tout[kk] = Tn[j];
                    collide<C>(g[j], dr[j], uu[j], vv[j], omega, fx, Gy, [&](int q, C v) { st(out + q * plane, v); });
                } else {
                    S *out = F + fi(lx, ly);
                    collide<C>(g[j], dr[j], uu[j], vv[j], omega, fx, Gy, [&](int q, C v) { st(out + q * PL, v); });
                }
            }
        }
        if (last) break;
        __syncthreads();
        // Exchange of the new populations and temperature.
        {
            const uint32_t tag = r.seq0 + (uint32_t)k + 1u;
            const uint32_t tag_t = (r.seq0 + (uint32_t)k) * (uint32_t)m + (uint32_t)m;
            uint64_t *slot = own + (size_t)(tag & 1u) * G::PACKETS * WORDS;
            C *To = T + cb * PL;
#pragma unroll
            for (int i = 0; i < NSF; i++)
                if (sf[i] >= 0) mail::post(slot, tid + i * BLOCK, F[sf[i]], tag ^ spoil);
            post_T(To, tag_t ^ spoil);
            // (both, one after the other's success or not: their first loads overlap)
            ok &= read(F, rf_at, rf_to, std::integral_constant<int, NRF>{}, tag, k);
            ok &= read(To, rt_at, rt_to, std::integral_constant<int, NRD>{}, tag_t, k);
            if (!ok) gave_up = 1;
        }
        __syncthreads();
        if (gave_up) {
            if (!ok) atomicOr(r.a.err, kErrTimeout);
            return;
        }
    }
}

// Tile shapes, smallest first: the host takes the first one whose tiles fit
// the SMs one per block.  Fewer nodes per SM mean a shorter step until the
// exchange dominates, so the smallest shape that fits is the fastest (the
// 64-column ones not always faster than one launch per step, see the host's
// resident_pays).  Where
// no shape fits, or only one whose registers spill, one launch per step is the
// faster (f32 64 x 40 tiles at 600^2: 9.2 us against 9.0; double-single 32 x 32
// at 320^2: 32.5 against 15.7; FP64 74 against 63), so the lists end there.
constexpr int kResShapes = 6;
template <class S> constexpr int res_shapes() { return sizeof(S) == 2 ? 6 : 5; }
template <class S, int I> struct ResConfig;
template <class S> struct ResConfig<S, 0> { using G = ResTile<S, 16, 8, 128, 64>; };
template <class S> struct ResConfig<S, 1> { using G = ResTile<S, 32, 8, 256, 96>; };
template <class S> struct ResConfig<S, 2> { using G = ResTile<S, 32, 16, 512, 96>; };
template <class S> struct ResConfig<S, 3> { using G = ResTile<S, 32, 32, 512, 128>; };
template <class S> struct ResConfig<S, 4> { using G = ResTile<S, 64, 32, 512, 128>; };
template <class S> struct ResConfig<S, 5> { using G = ResTile<S, 64, 40, 512, 128>; };
#define LBMFVM_RES_WIDE(S, QUAD)                                                     \
    template <> struct ResConfig<S, 0> { using G = ResTile<S, 8, 4, 32 * QUAD, 32>; }; \
    template <> struct ResConfig<S, 1> { using G = ResTile<S, 8, 8, 64, 32>; };    \
    template <> struct ResConfig<S, 2> { using G = ResTile<S, 16, 8, 128, 64>; };  \
    template <> struct ResConfig<S, 3> { using G = ResTile<S, 32, 8, 256, 96>; };  \
    template <> struct ResConfig<S, 4> { using G = ResTile<S, 32, 16, 256, 96>; };
LBMFVM_RES_WIDE(double, 4)
LBMFVM_RES_WIDE(dsf, 1)
#undef LBMFVM_RES_WIDE

}  // namespace lbmfvm_dev

namespace lbmfvm_fv {

// Geometry of resident shape i (0 .. kResShapes - 1; TW = 0: the type has none).
struct ResShape {
    int TW, TH;
    size_t mail_bytes;  // mailbox of one tile
};
template <class S>
ResShape resident_shape(int i);
// Blocks of the shape's kernel that fit an SM (its shared-memory limit set).
template <class S>
cudaError_t resident_prepare(int i, lbmfvm_dev::ResForm form, int *blocks_per_sm);
// Cooperative launch over `tiles` blocks.
template <class S>
cudaError_t resident_launch(int i, lbmfvm_dev::ResForm form, const lbmfvm_dev::ResArgs<S> &r, int tiles,
                            cudaStream_t stream);

}  // namespace lbmfvm_fv
