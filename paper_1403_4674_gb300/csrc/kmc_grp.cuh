// kmc_grp.cuh -- a group of G lanes per 16x16, 32x32 or 64x64 domain, state in
// shared memory for the whole launch.
//
// What bounds these lattices is the chain of real events of the busiest
// domains, one after another, with four hand-offs between neighbours per
// schedule.  One lane per domain (32 domain processes per warp) makes an
// event a chain of some 600 instructions of one thread, 1600-2100 cycles; a
// whole warp per domain pays a five-round scan and ten class counts by warp
// reductions, 1800 cycles.  Here a warp runs 32 / G domains of one colour and
// the lanes of a group split a domain's rows (RPL each) between them:
//   * every lane holds its rows and their bit-sliced count planes in registers
//     for the visit, and forms the class mask of its own rows only;
//   * every lane holds the class counts of all rows above its own (E) and of
//     the domain (T) as two words of five 12-bit fields, so the member's lane
//     is found by one comparison per lane, with no scan; it broadcasts the
//     site, four lanes find the classes of its four neighbours from the spins
//     in shared memory side by side, and every lane applies the same five
//     class moves to T and those of them that lie above its rows to E;
//   * the class rates follow from T in every lane alike; the next event of 32
//     drawn steps is found by one vote per G steps.
// The trajectory is the warp kernel's, decision for decision: step j of
// global phase np draws Philox {j, d, np_lo, np_hi} with the replica seed,
// target = (w0 | w1<<32) >> 1 against R' = sum_c n_c A_c, class = first c
// with target < C_c, member jj = (target - C_{c-1}) / A_c in row-major order.
//
// Measured, whole calls: 1024^2 at L_d = 32, k = 4, 200 schedules 3.26 -> 1.07
// ms (before: one lane per domain); 64^2 at L_d = 16, k = 1, 1000 schedules
// 9.58 -> 5.1 to 5.5 ms; 16 lattices of 256^2 at L_d = 16 in random colour order, 40
// schedules 1.25 -> 0.64 ms (before: one warp per domain).  ncu, 1024 domains
// of 32x32 at G = 32: 0.9 warps per scheduler, 28 % of the issue slots, 31 of
// 32 threads active, stalls led by fixed-latency waits (1.2 cycles per
// instruction) and the halo reads (0.65): the chain of dependent
// instructions is the bound, not issue, memory or shared-memory banks.
//
// Halos come from the neighbours' stamped edge words: in shared memory when
// the neighbour is in the same CTA, else in global memory (L2).
//
// Scope: every colour schedule, exponential and expected clocks, per-replica
// k, records at schedule endpoints or every colour pass.  Fixed-time visits
// and scores use the other kernels.
#pragma once

#include "kmc_tpdr.cuh"
#include "kmc_tpdr64.cuh"

namespace kmcdev {

template <int LD, int G> struct GrpGeo {
    static_assert((LD == 16 || LD == 32 || LD == 64) && LD % G == 0 && LD / G <= 4, "domain side, lanes per domain");
    static constexpr int RPL = LD / G;            // rows per lane (1, 2 or 4)
    static constexpr int DPW = 32 / G;            // domains per warp (a set)
    static constexpr int SLOTS = 32 / G;          // steps of a chunk of 32 per lane
    static constexpr uint32_t GM = (G == 32) ? 0xFFFFFFFFu : ((1u << (G & 31)) - 1u);
    using row_t = typename std::conditional<(LD > 32), uint64_t, uint32_t>::type;
    static constexpr row_t FULL = (LD == 64) ? (row_t)~0ull : (row_t)((1ull << LD) - 1ull);
    // shared memory of one domain (bytes): per-lane counts of the rows above
    // (lo, hi), acceptances A_c and their reciprocals floor((2^64 - 1) / A_c),
    // each lane's clock product since the open record began (mantissa,
    // exponent), the domain's counts (lo, hi), u32 g, d, k (0: no domain),
    // replica, the halo columns that the counts hold (W, E; bit y = row y), the
    // domain's W and E columns, the rows after the N halo row and before the S
    // one (16 bytes from RING on hold the N halo row last), stamped edge words,
    // counters (hash, flips, steps, clock mantissa and exponent), the open
    // record (record | steps << 32, bonds | mag << 32), addresses of the
    // neighbours' edge words, seed, the events of the chunk (step | class << 5 |
    // site << 9)
    static constexpr int E = 0, AT = E + 16 * G, MR = AT + 80, CLK = MR + 80, T = CLK + 16 * G, META = T + 16,
                         HALO = META + 16, COLS = HALO + 16, RING = COLS + 16, ROWS = RING + 16,
                         EDGE = ROWS + (LD + 1) * (int)sizeof(row_t) + (LD == 64 ? 0 : 8 - (int)sizeof(row_t)),
                         CTR = EDGE + 64, OBS = CTR + 40, NBP = OBS + 16, SEED = NBP + 32, EV = SEED + 8, RAW = EV + 128;
    static_assert(EDGE % 8 == 0 && ROWS % 16 == 0, "aligned words");
    // an odd multiple of 16 bytes: the groups' words fall into different banks
    static constexpr int BYTES = ((RAW + 15) / 16 | 1) * 16;
};

// Class moves as differences of the packed counts {lo, hi}: entries dir * 10 +
// c: a neighbour of class c gains (dir 0) or loses (dir 1) an up neighbour;
// 20: no neighbour there; 21 + c: the site itself, of class c, flips.
constexpr int GRP_MOVES = 31;
constexpr int GRP_TABLE_BYTES = GRP_MOVES * 16;

template <int LD, int G> __host__ __device__ constexpr int grp_domain_bytes() { return GrpGeo<LD, G>::BYTES; }

// Bit offset of class c's field: down spins (c < 5) in reverse order, so that
// the two classes that can hold a whole domain (all down, all up) take the
// top field, which has 16 bits.
__host__ __device__ constexpr int grp_shift(int c) { return 12 * (c < 5 ? 4 - c : c - 5); }

__device__ __forceinline__ uint64_t ld_volatile_any(const uint64_t *p)
{
    uint64_t v;
    asm volatile("ld.volatile.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Position of the rr-th (0-based) set bit; rr < popc(w).
__device__ __forceinline__ int grp_select(uint32_t w, uint32_t rr) { return tpdr_select(w, rr); }
__device__ __forceinline__ int grp_select(uint64_t w, uint32_t rr)
{
    const uint32_t lo = (uint32_t)w, n = (uint32_t)__popc(lo);
    const bool up = rr >= n;
    return (up ? 32 : 0) + tpdr_select(up ? (uint32_t)(w >> 32) : lo, up ? rr - n : rr);
}

// Persistent kernel.  P.max_rt sets per warp; P.slot_g holds DPW domain ids
// per set (0xFFFFFFFF: none), P.cta_col_off the colour of each set (4: none),
// P.slot_nb four neighbours per domain (1 << 31 | slot in this CTA, or the
// global domain id).
template <int LD, int G, bool EXPO>
__global__ void __launch_bounds__(512, 1) grp_kernel(const RunParams P)
{
    using Q = GrpGeo<LD, G>;
    using row_t = typename Q::row_t;
    constexpr int RPL = Q::RPL, DPW = Q::DPW, SLOTS = Q::SLOTS;
    constexpr row_t FULL = Q::FULL;
    extern __shared__ __align__(16) uint8_t smem[];
    ulonglong2 *moves = reinterpret_cast<ulonglong2 *>(smem);
    uint8_t *domains = smem + GRP_TABLE_BYTES;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int gl = lane & (G - 1), grp = lane / G, gbase = lane - gl; // lane in its group, group, the group's first lane
    const int y0 = gl * RPL;                                          // the lane's first row
    const int ns = P.max_rt;
    const int wg = blockIdx.x * (blockDim.x >> 5) + wib;

    for (int i = threadIdx.x; i < GRP_MOVES; i += blockDim.x) {
        uint64_t d[2] = {0, 0};
        if (i < 20) {
            const int c = i % 10, to = (i < 10) ? c + 1 : c - 1;
            if (to >= 0 && to / 5 == c / 5 && to < 10) d[c / 5] = (1ull << grp_shift(to)) - (1ull << grp_shift(c));
        } else if (i > 20) {
            const int c = i - 21;
            d[c / 5] = 0ull - (1ull << grp_shift(c));
            d[1 - c / 5] = 1ull << grp_shift(c < 5 ? c + 5 : c - 5);
        }
        moves[i] = make_ulonglong2(d[0], d[1]);
    }

    auto dom = [&](int s) -> uint8_t * { return domains + (size_t)((wib * ns + s) * DPW + grp) * Q::BYTES; };
    auto u64 = [&](uint8_t *b, int off) -> uint64_t & { return *reinterpret_cast<uint64_t *>(b + off); };
    auto u32 = [&](uint8_t *b, int off) -> uint32_t & { return *reinterpret_cast<uint32_t *>(b + off); };
    auto row = [&](uint8_t *b, int y) -> row_t & { return reinterpret_cast<row_t *>(b + Q::ROWS)[y]; };

    // ---- stage the domains: rows, counts with an all-down halo ----
    // (every lane of a group asks for its share of the domain's words at once)
    for (int s = 0; s < ns; ++s) {
        uint8_t *b = dom(s);
        const size_t slot = ((size_t)wg * ns + s) * DPW + grp;
        const uint32_t g = P.slot_g[slot];
        const bool has = g != 0xFFFFFFFFu;
        const uint32_t nb = P.slot_nb[slot * 4 + (gl & 3)];
        const uint32_t r = has ? P.dom_rep[g] : 0u;
        const uint8_t *tile = P.tiles + (size_t)(has ? g : 0u) * (LD * LD / 8);
        row_t S[RPL];
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
            S[i] = (LD == 64) ? (row_t) reinterpret_cast<const uint64_t *>(tile)[y0 + i]
                   : (LD == 32) ? (row_t) reinterpret_cast<const uint32_t *>(tile)[y0 + i]
                                : (row_t) reinterpret_cast<const uint16_t *>(tile)[y0 + i];
            if (!has) S[i] = 0;
        }
        const uint64_t *edges = P.edges + (size_t)(has ? g : 0u) * EDGE_WORDS, *ctr = P.dctr + (size_t)(has ? g : 0u) * DCTR_WORDS;
        const uint64_t edge = edges[gl & 7];
        const int cw = (gl == 0) ? DCTR_HASH : (gl == 1) ? DCTR_FLIPS : (gl == 2) ? DCTR_STEPS : (gl == 3) ? DCTR_CLKM : DCTR_CLKE;
        const uint64_t count = ctr[cw];
        const uint64_t seed = P.rep_seed[r];
        const uint32_t k = (uint32_t)P.rep_k[r], doff = P.rep_dom_off[r];
        for (int c = gl; c < 10; c += G) {
            u64(b, Q::AT + 8 * c) = P.rep_A[(size_t)r * RATE_WORDS + c];
            u64(b, Q::MR + 8 * c) = P.rep_A[(size_t)r * RATE_WORDS + RATE_RECIP + c];
        }
#pragma unroll
        for (int i = 0; i < RPL; ++i) row(b, y0 + i) = S[i];
        if (gl == 0) row(b, -1) = row(b, LD) = 0;
        if (gl < 8) u64(b, Q::EDGE + 8 * gl) = has ? edge : 0ull;
        if (gl < 5) u64(b, Q::CTR + 8 * gl) = count;
        u64(b, Q::CLK + 16 * gl) = 1ull << 63;
        u64(b, Q::CLK + 16 * gl + 8) = 0;
        if (gl < 4) {
            // the neighbour's facing edge (N: its S row, S: its N row, W: its E
            // column, E: its W column); bit 0 of the address: in this CTA
            const int facing = gl ^ 1;
            uint64_t a = 0;
            if (has)
                a = (nb & 0x80000000u)
                        ? (uint64_t)(domains + (size_t)(nb & 0x7FFFFFFFu) * Q::BYTES + Q::EDGE + 16 * facing) | 1ull
                        : (uint64_t)(P.edges + (size_t)nb * EDGE_WORDS + 2 * facing);
            u64(b, Q::NBP + 8 * gl) = a;
        }
        __syncwarp();
        uint64_t lo = 0, hi = 0, cW = 0, cE = 0;
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
            const int y = y0 + i;
            const row_t U = row(b, y - 1), D = row(b, y + 1);
            const row_t Wn = (row_t)(S[i] << 1) & FULL, En = (row_t)(S[i] >> 1);
            const row_t s1 = U ^ D, c1 = U & D, s2 = Wn ^ En, c2 = Wn & En, t0 = s1 & s2;
            const row_t b0 = s1 ^ s2, b1 = c1 ^ c2 ^ t0, b2 = (c1 & c2) | (c1 & t0) | (c2 & t0);
            for (int q = 0; q < 5; ++q) {
                const row_t m = (row_t)(((q & 4) ? b2 : ~b2) & ((q & 2) ? b1 : ~b1) & ((q & 1) ? b0 : ~b0)) & FULL;
                lo += (uint64_t)popc_row((row_t)(m & ~S[i])) << grp_shift(q);
                hi += (uint64_t)popc_row((row_t)(m & S[i])) << grp_shift(5 + q);
            }
            cW |= (uint64_t)(S[i] & 1u) << y;
            cE |= (uint64_t)((S[i] >> (LD - 1)) & 1u) << y;
        }
        uint64_t ilo = lo, ihi = hi;
#pragma unroll
        for (int off = 1; off < G; off <<= 1) {
            const uint64_t a = __shfl_up_sync(FULL_WARP, ilo, off, G), c = __shfl_up_sync(FULL_WARP, ihi, off, G);
            ilo += (gl >= off) ? a : 0ull;
            ihi += (gl >= off) ? c : 0ull;
            cW |= __shfl_xor_sync(FULL_WARP, cW, off);
            cE |= __shfl_xor_sync(FULL_WARP, cE, off);
        }
        u64(b, Q::E + 16 * gl) = ilo - lo;
        u64(b, Q::E + 16 * gl + 8) = ihi - hi;
        if (gl == G - 1) {
            u64(b, Q::T) = ilo;
            u64(b, Q::T + 8) = ihi;
        }
        if (gl == 0) {
            u64(b, Q::COLS) = cW;
            u64(b, Q::COLS + 8) = cE;
            u64(b, Q::HALO) = u64(b, Q::HALO + 8) = 0;
            u64(b, Q::SEED) = seed;
            *reinterpret_cast<uint4 *>(b + Q::META) = make_uint4(g, has ? g - doff : 0u, has ? k : 0u, r);
            u64(b, Q::OBS) = (uint64_t)NO_RECORD;
            u64(b, Q::OBS + 8) = 0;
        }
        __syncwarp();
    }
    __syncthreads(); // the edge words of the CTA's domains are in place

    // The group's clock product since the record began, joined over its lanes
    // (each lane multiplies the variates of its own steps).  A step takes 1.44
    // off the exponent on average, and without records a launch's steps are
    // one product: past 1.49e9 steps of a domain it leaves 32 bits.
    auto joined_clock = [&](uint8_t *b, uint64_t &m, int64_t &e) {
        m = u64(b, Q::CLK + 16 * gl);
        e = (int64_t)u64(b, Q::CLK + 16 * gl + 8);
#pragma unroll
        for (int off = 1; off < G; off <<= 1) {
            const uint64_t m2 = __shfl_xor_sync(FULL_WARP, m, off);
            const int64_t e2 = __shfl_xor_sync(FULL_WARP, (long long)e, off);
            int up = 0;
            mant_mul32(m, up, m2, 0);
            e += e2 + up;
        }
        u64(b, Q::CLK + 16 * gl) = 1ull << 63;
        u64(b, Q::CLK + 16 * gl + 8) = 0;
    };
    // Close the open record of the group's domain: its sums go to the replica's
    // record (records past the launch's last one are dropped), its clock
    // product into the domain's clock.  Called by the whole warp.
    auto flush = [&](uint8_t *b) {
        uint64_t m = 1ull << 63;
        int64_t e = 0;
        if (EXPO) joined_clock(b, m, e);
        const bool mine = gl == 0 && u32(b, Q::META) != 0xFFFFFFFFu;
        const uint64_t o0 = u64(b, Q::OBS), o1 = u64(b, Q::OBS + 8);
        const uint32_t o = (uint32_t)o0;
        const bool on = mine && o != NO_RECORD && (int64_t)o < P.n_obs;
        double dt = 0.0;
        if (mine && EXPO) {
            uint64_t cm = u64(b, Q::CTR + 24);
            int64_t ce = (int64_t)u64(b, Q::CTR + 32);
            mant_mul(cm, ce, m, e);
            u64(b, Q::CTR + 24) = cm;
            u64(b, Q::CTR + 32) = (uint64_t)ce;
        }
        if (on)
            dt = EXPO ? domain_time(true, m, e, 0, P.lambda) : __ddiv_rn((double)(uint32_t)(o0 >> 32), P.lambda);
        // the set's domains are one replica's and share the record: one sum
        int bonds = on ? (int)(uint32_t)o1 : 0, mag = on ? (int)(uint32_t)(o1 >> 32) : 0;
#pragma unroll
        for (int off = G; off < 32; off <<= 1) {
            dt += __shfl_xor_sync(FULL_WARP, dt, off);
            bonds += __shfl_xor_sync(FULL_WARP, bonds, off);
            mag += __shfl_xor_sync(FULL_WARP, mag, off);
        }
        if (on && lane == 0) {
            unsigned long long *acc = P.obs_acc + ((size_t)o * P.n_rep + u32(b, Q::META + 12)) * OBS_WORDS;
            if (bonds != 0) atomicAdd(&acc[0], (unsigned long long)(long long)bonds);
            if (mag != 0) atomicAdd(&acc[1], (unsigned long long)(long long)mag);
            atomicAdd(reinterpret_cast<double *>(&acc[2]), dt);
        }
        __syncwarp();
    };

    const int nph = (P.schedule == SCHED_PALINDROME) ? 8 : 4;
    unsigned long long polls = 0; // halo re-reads of the warp (profiling)
    bool ok = true;

    // this lane's neighbour of an event's site (W, E, N, S by gl % 4), the edge
    // it publishes (lanes 0, 1, 2: N, W, E; the last lane: S) and the halo word
    // it polls (two halves per edge at 64 columns)
    const int dx = (gl & 2) ? 0 : (gl & 1) ? 1 : -1, dy = (gl & 2) ? ((gl & 1) ? 1 : -1) : 0;
    const int pub = (gl == 0) ? EDGE_N : (gl == 1) ? EDGE_W : (gl == 2) ? EDGE_E : (gl == G - 1) ? EDGE_S : -1;
    const int side = (LD == 64) ? (gl & 7) >> 1 : gl & 3, half = (LD == 64) ? gl & 1 : 0;

    // One visit of set s: nf fused phases from phase np0 on, for which the
    // neighbours' visit counts have to be at least needNS and needWE.
    auto visit = [&](int s, uint64_t np0, int nf, uint32_t needNS, uint32_t needWE, uint32_t after, int64_t o) {
        uint8_t *b = dom(s);
        const uint4 meta = *reinterpret_cast<const uint4 *>(b + Q::META);
        const uint32_t d = meta.y;
        const int k = (int)meta.z;
        const int total = nf * k;
        const uint64_t seed = u64(b, Q::SEED);
        const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
        const int smax = (int)__reduce_max_sync(FULL_WARP, (unsigned)total);

        // ---- what does not depend on the halo: the draws of the first 32
        // steps, rows, planes with the halo the counts hold, counts ----
        // lane gl draws steps base + gl, base + G + gl, ...: targets (~0 past
        // the last step), clock variates into the lane's product
        uint64_t tg[SLOTS];
        uint64_t vM = 1ull << 63;
        int vE = 0;
        auto draw = [&](int base) {
#pragma unroll
            for (int q = 0; q < SLOTS; ++q) {
                tg[q] = ~0ull;
                const int st = base + q * G + gl;
                if (base + q * G < smax && st < total) {
                    const int f = st >= k ? 1 : 0; // at most two phases fuse
                    const uint64_t np = np0 + (uint64_t)f;
                    const uint4 w = philox4x32_10(
                        make_uint4((uint32_t)(st - (f ? k : 0)), d, (uint32_t)np, (uint32_t)(np >> 32) & 0xFFFFFFu), key);
                    tg[q] = (((uint64_t)w.y << 32) | w.x) >> 1;
                    if (EXPO) {
                        const uint64_t V = ((((uint64_t)w.w << 32) | w.z) >> 11) + 1ull;
                        const int z = __clzll((long long)V);
                        mant_mul32(vM, vE, V << z, 10 - z);
                    }
                }
            }
        };
        draw(0);
        // the lane's rows y0 .. y0 + RPL - 1 and their up-neighbour counts b2 b1 b0
        row_t S[RPL], b0[RPL], b1[RPL], b2[RPL];
        uint64_t hW = u64(b, Q::HALO), hE = u64(b, Q::HALO + 8);
        {
            row_t R[RPL + 2];
#pragma unroll
            for (int i = 0; i < RPL + 2; ++i) R[i] = row(b, y0 - 1 + i);
#pragma unroll
            for (int i = 0; i < RPL; ++i) {
                S[i] = R[i + 1];
                const row_t U = R[i], D = R[i + 2];
                const row_t Wn = ((row_t)(S[i] << 1) | (row_t)((hW >> (y0 + i)) & 1ull)) & FULL;
                const row_t En = (row_t)(S[i] >> 1) | ((row_t)((hE >> (y0 + i)) & 1ull) << (LD - 1));
                const row_t s1 = U ^ D, c1 = U & D, s2 = Wn ^ En, c2 = Wn & En, t0 = s1 & s2;
                b0[i] = s1 ^ s2;
                b1[i] = c1 ^ c2 ^ t0;
                b2[i] = (c1 & c2) | (c1 & t0) | (c2 & t0);
            }
        }
        ulonglong2 E = *reinterpret_cast<const ulonglong2 *>(b + Q::E + 16 * gl);
        ulonglong2 T = *reinterpret_cast<const ulonglong2 *>(b + Q::T);

        // ---- the halo: lane gl reads one stamped word of one neighbour ----
        constexpr int HW = (LD == 64) ? 8 : 4;
        uint64_t w = 0;
        {
            const uint64_t *src = reinterpret_cast<const uint64_t *>(u64(b, Q::NBP + 8 * side) & ~1ull) + half;
            const uint32_t need = side < 2 ? needNS : needWE;
            bool ready = k == 0;
            if (!ready) {
                w = ld_volatile_any(src);
                ready = (uint32_t)(w >> 32) >= need;
            }
            if (!__all_sync(FULL_WARP, ready)) {
                const uint64_t t0 = global_ns();
                unsigned it = 0;
                while (true) {
                    if (!ready) {
                        w = ld_volatile_any(src);
                        ready = (uint32_t)(w >> 32) >= need;
                    }
                    ++polls;
                    if (__all_sync(FULL_WARP, ready)) break;
                    if ((++it & 63u) == 0) {
                        const bool late = global_ns() - t0 > P.bar_limit_ns;
                        const bool quit = late || *(volatile int *)P.err != 0;
                        if (__any_sync(FULL_WARP, quit)) {
                            if (late) atomicCAS(P.err, 0, ERR_TIMEOUT);
                            ok = false;
                            break;
                        }
                    }
                }
                if (!ok) return;
            }
        }
        // ---- sites whose halo bits changed since the counts were built:
        // each gains or loses an up neighbour ----
        {
            auto word = [&](int q) { return __shfl_sync(FULL_WARP, (uint32_t)w, gbase + q); };
            row_t nN, nS;
            uint64_t nW, nE;
            if (HW == 8) {
                nN = (row_t)((uint64_t)word(0) | ((uint64_t)word(1) << 32));
                nS = (row_t)((uint64_t)word(2) | ((uint64_t)word(3) << 32));
                // a column's halves hold its even and its odd rows
                const uint64_t sp = t64_spread((uint32_t)w);
                nW = __shfl_sync(FULL_WARP, sp, gbase + 4) | (__shfl_sync(FULL_WARP, sp, gbase + 5) << 1);
                nE = __shfl_sync(FULL_WARP, sp, gbase + 6) | (__shfl_sync(FULL_WARP, sp, gbase + 7) << 1);
            } else {
                nN = word(0);
                nS = word(1);
                nW = word(2);
                nE = word(3);
            }
            const row_t oN = row(b, -1), oS = row(b, LD);
            const bool same = k == 0 || (nN == oN && nS == oS && nW == hW && nE == hE);
            if (!__all_sync(FULL_WARP, same)) {
                const uint64_t mine = (1ull << RPL) - 1ull;
                row_t tN = (gl == 0) ? nN ^ oN : (row_t)0, tS = (gl == G - 1) ? nS ^ oS : (row_t)0;
                uint32_t tWE = (uint32_t)(((nW ^ hW) >> y0) & mine) | ((uint32_t)(((nE ^ hE) >> y0) & mine) << RPL);
                if (k == 0) {
                    tN = tS = 0;
                    tWE = 0;
                }
                uint64_t dlo = 0, dhi = 0;
                while (__any_sync(FULL_WARP, (tN | tS) != 0 || tWE != 0)) {
                    if ((tN | tS) != 0 || tWE != 0) {
                        int i, col;
                        bool up;
                        if (tWE) {
                            const int z = __ffs((int)tWE) - 1;
                            tWE &= tWE - 1;
                            const bool east = z >= RPL;
                            i = east ? z - RPL : z;
                            col = east ? LD - 1 : 0;
                            up = ((east ? nE : nW) >> (y0 + i)) & 1ull;
                        } else if (tN) {
                            col = __ffsll((long long)tN) - 1;
                            tN &= tN - 1;
                            i = 0;
                            up = (nN >> col) & 1u;
                        } else {
                            col = __ffsll((long long)tS) - 1;
                            tS &= tS - 1;
                            i = RPL - 1;
                            up = (nS >> col) & 1u;
                        }
                        const row_t bit = (row_t)1 << col, L = up ? (row_t)0 : (row_t)~(row_t)0;
                        int c = 0;
#pragma unroll
                        for (int r = 0; r < RPL; ++r) {
                            const row_t m = (r == i) ? bit : (row_t)0;
                            c += ((S[r] & m) ? 5 : 0) + ((b0[r] & m) ? 1 : 0) + ((b1[r] & m) ? 2 : 0) + ((b2[r] & m) ? 4 : 0);
                            const row_t c0 = (b0[r] ^ L) & m;
                            b0[r] ^= m;
                            const row_t c1 = (b1[r] ^ L) & c0;
                            b1[r] ^= c0;
                            b2[r] ^= c1;
                        }
                        const ulonglong2 mv = moves[(up ? 0 : 10) + c];
                        dlo += mv.x;
                        dhi += mv.y;
                    }
                }
                uint64_t ilo = dlo, ihi = dhi;
#pragma unroll
                for (int off = 1; off < G; off <<= 1) {
                    const uint64_t a = __shfl_up_sync(FULL_WARP, ilo, off, G), c = __shfl_up_sync(FULL_WARP, ihi, off, G);
                    ilo += (gl >= off) ? a : 0ull;
                    ihi += (gl >= off) ? c : 0ull;
                }
                E.x += ilo - dlo;
                E.y += ihi - dhi;
                T.x += __shfl_sync(FULL_WARP, ilo, G - 1, G);
                T.y += __shfl_sync(FULL_WARP, ihi, G - 1, G);
                hW = nW;
                hE = nE;
                __syncwarp();
                if (k != 0) {
                    row(b, -1) = nN;
                    row(b, LD) = nS;
                    u64(b, Q::HALO) = nW;
                    u64(b, Q::HALO + 8) = nE;
                }
                __syncwarp();
            }
        }

        // cumulative class rates C_c = sum_{c' <= c} n_c' A_c'; C[9] = R' (the
        // acceptances in registers where the rows leave room)
        uint64_t C[10], A[10];
        if (RPL * (int)sizeof(row_t) <= 8) {
#pragma unroll
            for (int c = 0; c < 10; ++c) A[c] = u64(b, Q::AT + 8 * c);
        }
        auto rates = [&]() {
            uint64_t W[10];
#pragma unroll
            for (int c = 0; c < 10; ++c) {
                const int sh = grp_shift(c);
                const uint32_t n = (sh == 48) ? (uint32_t)((c < 5 ? T.x : T.y) >> 48) : (uint32_t)((c < 5 ? T.x : T.y) >> sh) & 0xFFFu;
                W[c] = (uint64_t)n * (RPL * (int)sizeof(row_t) <= 8 ? A[c] : u64(b, Q::AT + 8 * c));
            }
            const uint64_t s23 = W[2] + W[3], s45 = W[4] + W[5], s67 = W[6] + W[7], s89 = W[8] + W[9];
            C[0] = W[0];
            C[1] = W[0] + W[1];
            C[2] = C[1] + W[2];
            C[3] = C[1] + s23;
            C[4] = C[3] + W[4];
            C[5] = C[3] + s45;
            C[6] = C[5] + W[6];
            C[7] = C[5] + s67;
            C[8] = C[7] + W[8];
            C[9] = C[7] + s89;
        };
        rates();
        row_t colW = (row_t)u64(b, Q::COLS), colE = (row_t)u64(b, Q::COLS + 8);
        bool corrupt = false; // counts and spins disagreed at some event

        // What the events add to the event hash, the bond sum and the
        // magnetisation is worked off from the list of the chunk's events,
        // after the visit's edges are published.
        uint64_t H = u64(b, Q::CTR);
        uint32_t ne = 0, flips = 0; // events of the chunk, of the visit
        int dbonds = 0, dmag = 0;
        auto work_off = [&](int base) {
            __syncwarp();
            const int most = (int)__reduce_max_sync(FULL_WARP, ne);
            for (int i = 0; i < most; ++i) {
                const uint32_t e = u32(b, Q::EV + 4 * i);
                const int sg = base + (int)(e & 31u), c = (int)((e >> 5) & 15u), f = sg >= k ? 1 : 0;
                const uint64_t np = np0 + (uint64_t)f;
                const uint64_t h = (H ^ ((np << 32) | ((uint64_t)(sg - (f ? k : 0)) << 16) | (uint64_t)(e >> 9))) * HASH_PRIME;
                const bool act = i < (int)ne;
                H = act ? h : H;
                // flipping spin s with neighbour sum 2 q - 4 changes the bond sum
                // by -2 s (2 q - 4) and the magnetisation by -2 s
                const int g2 = act ? (c < 5 ? 2 : -2) : 0;
                dbonds += g2 * (2 * (c < 5 ? c : c - 5) - 4);
                dmag += g2;
            }
            flips += ne;
            ne = 0;
            __syncwarp();
        };

        for (int base = 0; base < smax; base += 32) {
            if (base > 0) {
                work_off(base - 32);
                draw(base);
            }
            uint32_t left = 0xFFFFFFFFu; // steps of the chunk not passed yet
            while (true) {
                // the group's next step that may have target < R' (by the high
                // words): bit q G + l is lane l's q-th step
                uint32_t m = 0;
#pragma unroll
                for (int q = 0; q < SLOTS; ++q) {
                    const uint32_t v = __ballot_sync(FULL_WARP, (uint32_t)(tg[q] >> 32) <= (uint32_t)(C[9] >> 32));
                    m |= ((v >> gbase) & Q::GM) << ((q * G) & 31);
                }
                m &= left;
                if (!__any_sync(FULL_WARP, m != 0)) break;
                const int st = m ? __ffs((int)m) - 1 : 0;
                left = m ? (0xFFFFFFFEu << st) : 0u;
                uint64_t t = tg[0];
#pragma unroll
                for (int q = 1; q < SLOTS; ++q) t = (st >= q * G) ? tg[q] : t;
                t = __shfl_sync(FULL_WARP, t, gbase + (st & (G - 1)));
                const bool act = m != 0 && t < C[9]; // a real event
                // class: the first c with t < C_c
                int c = 0;
                uint64_t Cprev = 0;
#pragma unroll
                for (int cc = 0; cc < 9; ++cc) {
                    const bool past = t >= C[cc];
                    c += past ? 1 : 0;
                    Cprev = past ? C[cc] : Cprev;
                }
                const uint64_t Ac = u64(b, Q::AT + 8 * c), Mc = u64(b, Q::MR + 8 * c);
                // exact jj = floor((t - C_{c-1}) / A_c) < n_c: the high word of
                // (t - C_{c-1}) floor((2^64 - 1) / A_c) is jj or jj - 1
                const uint64_t x = t - Cprev;
                uint32_t jj = (uint32_t)__umul64hi(x, Mc);
                jj = (x - (uint64_t)jj * Ac >= Ac) ? jj + 1u : jj;
                const bool up = c >= 5;
                const int qc = up ? c - 5 : c;
                const int sh = 12 * (up ? qc : 4 - qc);
                // members in this lane's rows, in row-major order
                const row_t UP = up ? (row_t)0 : (row_t)~(row_t)0, Q2 = (qc & 4) ? (row_t)0 : (row_t)~(row_t)0,
                            Q1 = (qc & 2) ? (row_t)0 : (row_t)~(row_t)0, Q0 = (qc & 1) ? (row_t)0 : (row_t)~(row_t)0;
                row_t mk[RPL];
                uint32_t pf[RPL];
#pragma unroll
                for (int i = 0; i < RPL; ++i) {
                    mk[i] = (S[i] ^ UP) & (b2[i] ^ Q2) & (b1[i] ^ Q1) & (b0[i] ^ Q0) & FULL;
                    pf[i] = (uint32_t)popc_row(mk[i]) + (i ? pf[i ? i - 1 : 0] : 0u);
                }
                const uint32_t rem = jj - ((uint32_t)((up ? E.y : E.x) >> sh) & 0xFFFu);
                const uint32_t wins = (__ballot_sync(FULL_WARP, rem < pf[RPL - 1]) >> gbase) & Q::GM;
                // the member's row and column (computed by every lane, taken
                // from the one that owns it)
                int yi = 0;
                uint32_t before = 0;
                row_t mask = mk[0];
#pragma unroll
                for (int i = 1; i < RPL; ++i) {
                    const bool past = rem >= pf[i - 1];
                    yi = past ? i : yi;
                    before = past ? pf[i - 1] : before;
                    mask = past ? mk[i] : mask;
                }
                uint32_t msg = (uint32_t)(grp_select(mask, rem - before) & (LD - 1)) | ((uint32_t)(y0 + yi) << 6);
                msg = __shfl_sync(FULL_WARP, msg, gbase + (wins ? __ffs((int)wins) - 1 : 0));
                const int col = (int)(msg & 63u), y = (int)(msg >> 6);
                // the class of this lane's neighbour of the site, from the spins
                uint32_t move;
                {
                    const int xx = col + dx, yy = y + dy;
                    const bool in = act && (unsigned)xx < (unsigned)LD && (unsigned)yy < (unsigned)LD;
                    const int xi = xx & (LD - 1), yv = yy & (LD - 1);
                    constexpr int W32 = LD == 64 ? 2 : 1;
                    const uint32_t *r32 = reinterpret_cast<const uint32_t *>(b + Q::ROWS);
                    auto bit = [&](int bx, int by) { return (r32[by * W32 + (bx >> 5)] >> (bx & 31)) & 1u; };
                    const uint32_t wb = (xi > 0) ? bit(xi - (xi > 0 ? 1 : 0), yv) : (uint32_t)(hW >> yv) & 1u;
                    const uint32_t eb = (xi < LD - 1) ? bit(xi + (xi < LD - 1 ? 1 : 0), yv) : (uint32_t)(hE >> yv) & 1u;
                    const uint32_t cl = 5u * bit(xi, yv) + wb + eb + bit(xi, yv - 1) + bit(xi, yv + 1);
                    // a spin that flips up gives its neighbours an up neighbour
                    move = in ? (up ? 10u : 0u) + cl : 20u;
                }
                const ulonglong2 mY = moves[act ? 21 + c : 20];
                const ulonglong2 mW = moves[__shfl_sync(FULL_WARP, move, gbase)], mE = moves[__shfl_sync(FULL_WARP, move, gbase + 1)],
                                 mN = moves[__shfl_sync(FULL_WARP, move, gbase + 2)],
                                 mS = moves[__shfl_sync(FULL_WARP, move, gbase + 3)];
                __syncwarp(); // every lane has read the spins
                corrupt |= act && wins == 0;
                const uint64_t ylo = mY.x + mW.x + mE.x, yhi = mY.y + mW.y + mE.y;
                T.x += ylo + (mN.x + mS.x);
                T.y += yhi + (mN.y + mS.y);
                rates();
                E.x += (y < y0 ? ylo : 0ull) + (y <= y0 ? mN.x : 0ull) + (y + 1 < y0 ? mS.x : 0ull);
                E.y += (y < y0 ? yhi : 0ull) + (y <= y0 ? mN.y : 0ull) + (y + 1 < y0 ? mS.y : 0ull);
                const row_t bit = act ? (row_t)1 << col : (row_t)0, mh = ((row_t)(bit << 1) | (row_t)(bit >> 1)) & FULL;
                const row_t L = up ? (row_t)~(row_t)0 : (row_t)0;
                const int at = y - y0;
#pragma unroll
                for (int i = 0; i < RPL; ++i) {
                    const row_t mm = (i == at) ? mh : (i == at - 1 || i == at + 1) ? bit : (row_t)0;
                    if (i == at) {
                        S[i] ^= bit;
                        row(b, y) = S[i];
                    }
                    const row_t c0 = (b0[i] ^ L) & mm;
                    b0[i] ^= mm;
                    const row_t c1 = (b1[i] ^ L) & c0;
                    b1[i] ^= c0;
                    b2[i] ^= c1;
                }
                if (col == 0) colW ^= act ? (row_t)1 << y : (row_t)0;
                if (col == LD - 1) colE ^= act ? (row_t)1 << y : (row_t)0;
                if (act) u32(b, Q::EV + 4 * (int)ne) = (uint32_t)st | ((uint32_t)c << 5) | ((uint32_t)(y * LD + col) << 9);
                ne += act ? 1u : 0u;
                __syncwarp(); // the flipped spin is in place
            }
        }
        if (corrupt) atomicCAS(P.err, 0, ERR_INTERNAL);

        // ---- edges first (neighbours wait for them), then the state ----
        if (k != 0) {
            if (pub >= 0) {
                const uint64_t cnt = (uint64_t)after << 32;
                uint64_t v = (pub == EDGE_N) ? (uint64_t)S[0] : (pub == EDGE_W) ? (uint64_t)colW : (pub == EDGE_E) ? (uint64_t)colE : (uint64_t)S[RPL - 1];
                if (LD == 64 && (pub == EDGE_W || pub == EDGE_E)) v = t64_col_to_edge(v);
                volatile uint64_t *own = reinterpret_cast<volatile uint64_t *>(b + Q::EDGE) + 2 * pub;
                const uint64_t v0 = cnt | (uint32_t)v, v1 = cnt | (uint32_t)(v >> 32);
                own[0] = v0;
                if (LD == 64) own[1] = v1;
                // (this edge's reader is the neighbour on its side)
                if ((u64(b, Q::NBP + 8 * pub) & 1ull) == 0) {
                    uint64_t *out = P.edges + (size_t)meta.x * EDGE_WORDS + 2 * pub;
                    st_cg(out, v0);
                    if (LD == 64) st_cg(out + 1, v1);
                }
            }
            // (each word by its owner, or the same value by every lane of the group)
            *reinterpret_cast<ulonglong2 *>(b + Q::E + 16 * gl) = E;
            *reinterpret_cast<ulonglong2 *>(b + Q::T) = T;
            u64(b, Q::COLS) = (uint64_t)colW;
            u64(b, Q::COLS + 8) = (uint64_t)colE;
        }
        work_off((smax - 1) / 32 * 32);
        if (P.n_obs > 0 && __any_sync(FULL_WARP, k != 0 && (int64_t)(uint32_t)u64(b, Q::OBS) != o)) {
            // (every domain of the warp sees the same phases: all change record together)
            flush(b);
            u64(b, Q::OBS) = (uint64_t)(uint32_t)o;
            u64(b, Q::OBS + 8) = 0;
            __syncwarp();
        }
        if (EXPO) {
            uint64_t m = u64(b, Q::CLK + 16 * gl);
            mant_mul32(m, vE, vM, 0);
            u64(b, Q::CLK + 16 * gl) = m;
            u64(b, Q::CLK + 16 * gl + 8) += (uint64_t)(int64_t)vE;
        }
        const uint64_t fl = u64(b, Q::CTR + 8), nst = u64(b, Q::CTR + 16), o0 = u64(b, Q::OBS), o1 = u64(b, Q::OBS + 8);
        __syncwarp();
        u64(b, Q::CTR) = H;
        u64(b, Q::CTR + 8) = fl + flips;
        u64(b, Q::CTR + 16) = nst + (uint64_t)total;
        u64(b, Q::OBS) = (uint64_t)(uint32_t)o0 | ((uint64_t)((uint32_t)(o0 >> 32) + (uint32_t)total) << 32);
        u64(b, Q::OBS + 8) = (uint64_t)(uint32_t)((int)(uint32_t)o1 + dbonds) |
                             ((uint64_t)(uint32_t)((int)(uint32_t)(o1 >> 32) + dmag) << 32);
        __syncwarp();
    };

    uint32_t setcol = 0; // the colours of the warp's sets, four bits each
    for (int s = 0; s < ns; ++s) setcol |= P.cta_col_off[(size_t)wg * ns + s] << (4 * s);
    // The warp walks its own phases only: the phases p of a schedule that have
    // one of its sets' colours, and for each the visits that every colour's
    // domains have completed before it, in closed form.  Two phases of one
    // colour in a row are one visit (the palindrome's middle, and its ends
    // where two schedules meet) unless an observation falls between them.
    // With random orders every replica has its own order of the four colours in
    // every schedule; a colour's domains then complete one visit per schedule.
    const bool pal = P.schedule == SCHED_PALINDROME, fuse = pal && !P.obs_pass, perm = P.schedule == SCHED_RANDOM_PERM;
    uint32_t phases = 0;
    for (int p = 0; p < nph; ++p)
        for (int s = 0; s < ns; ++s)
            if (perm || (int)((setcol >> (4 * s)) & 15u) == fixed_colour(P.schedule, p)) phases |= 1u << p;
    if (fuse) phases &= ~(1u << 4);
    uint32_t rec = 0;                     // records completed by whole schedules
    int32_t until = P.obs_every;          // schedules left before the next one
    bool joined = false;                  // phase 0 ran with the last schedule's phase 7
    for (int64_t nl = 0; nl < P.n_sched && ok; ++nl) {
        const uint32_t n32 = (uint32_t)nl;
        const bool ends = P.obs_every > 0 && !P.obs_pass && until == 1; // a record follows this schedule
        const bool join = fuse && !ends && nl + 1 < P.n_sched;
        const uint64_t n = (uint64_t)P.sched_begin + (uint64_t)nl;
        uint32_t orders = 0; // of the sets' replicas, a byte each
        if (perm)
            for (int s = 0; s < ns; ++s)
                orders |= perm_order(u64(domains + (size_t)((wib * ns + s) * DPW) * Q::BYTES, Q::SEED), n) << (8 * s);
        for (uint32_t rest = joined ? phases & ~1u : phases; rest != 0 && ok; rest &= rest - 1) {
            const int p = __ffs((int)rest) - 1;
            const int nf = (fuse && (p == 3 || (p == 7 && join))) ? 2 : 1;
            // the visit's changes belong to the first record at or after its pass
            const int64_t o = P.obs_pass ? (nl * nph + p) / P.obs_every : (int64_t)rec;
            for (int s = 0; s < ns && ok; ++s) {
                const int colour = (int)((setcol >> (4 * s)) & 15u);
                const uint32_t order = (orders >> (8 * s)) & 0xFFu;
                if (colour != (perm ? (int)((order >> (2 * p)) & 3u) : fixed_colour(P.schedule, p))) continue;
                // visits of colour c completed before phase p of schedule nl
                auto before = [&](int c) -> uint32_t {
                    if (perm) {
                        const uint32_t twice = (uint32_t)c * 0x55u, hit = ~(order ^ twice), // both bits set where order holds c
                            at = hit & (hit >> 1) & 0x55u;
                        return n32 + ((at & ((1u << (2 * p)) - 1u)) ? 1u : 0u);
                    }
                    if (!pal) return n32 + (p > c ? 1u : 0u);
                    if (!fuse) return 2 * n32 + (p > c ? 1u : 0u) + (p > 7 - c ? 1u : 0u);
                    if (c == 0) return n32 + rec + (p > 0 ? 1u : 0u);
                    if (c == 3) return n32 + (p > 3 ? 1u : 0u);
                    return 2 * n32 + (p > c ? 1u : 0u) + (p > 7 - c ? 1u : 0u);
                };
                // a neighbour across a row has colour ^ 2, across a column colour ^ 1
                visit(s, n * 8 + (uint64_t)p, nf, before(colour ^ 2) + (uint32_t)P.debug_extra,
                      before(colour ^ 1) + (uint32_t)P.debug_extra, before(colour) + 1, o);
            }
        }
        joined = join;
        if (P.obs_every > 0 && !P.obs_pass && --until == 0) {
            ++rec;
            until = P.obs_every;
        }
    }
    if (P.polls && lane == 0 && polls != 0) atomicAdd(P.polls, polls);
    __syncthreads();
    if (__any_sync(FULL_WARP, *(volatile int *)P.err != 0)) return; // (whole warps: records are closed by the warp)
    // write the domains back: tile, counters, open record
    for (int s = 0; s < ns; ++s) {
        uint8_t *b = dom(s);
        flush(b);
        const uint32_t g = u32(b, Q::META);
        if (g == 0xFFFFFFFFu) continue;
        uint8_t *tile = P.tiles + (size_t)g * (LD * LD / 8);
        for (int y = y0; y < y0 + RPL; ++y) {
            if (LD == 64) reinterpret_cast<uint64_t *>(tile)[y] = (uint64_t)row(b, y);
            else if (LD == 32) reinterpret_cast<uint32_t *>(tile)[y] = (uint32_t)row(b, y);
            else reinterpret_cast<uint16_t *>(tile)[y] = (uint16_t)row(b, y);
        }
        if (gl == 0) {
            uint64_t *ctr = P.dctr + (size_t)g * DCTR_WORDS;
            ctr[DCTR_HASH] = u64(b, Q::CTR);
            ctr[DCTR_FLIPS] = u64(b, Q::CTR + 8);
            ctr[DCTR_STEPS] = u64(b, Q::CTR + 16);
            ctr[DCTR_CLKM] = u64(b, Q::CTR + 24);
            ctr[DCTR_CLKE] = u64(b, Q::CTR + 32);
        }
    }
}

} // namespace kmcdev
