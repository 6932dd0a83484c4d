// kmc_tpd.cuh -- one thread per domain visit, for 8x8 domains.
//
// An 8x8 domain is one 64-bit word (row y at bits [8y, 8y+8), bit x = column
// x, the bit tile layout of the lattice kernels), so one thread can run a
// whole domain process (Sec. 2.2) in registers: the frozen halo is four
// 8-bit masks, the up-neighbour counts are three bit-sliced 64-bit planes,
// every class of App. A is a 64-bit mask, the cumulative class rates are ten
// 64-bit integers, and the n-fold way's member choice is a bit selection in
// one word.  A warp then runs 32 domain processes with no warp-collective
// operation at all, where the warp-per-domain kernel spends a whole warp
// (8 of its lanes holding rows) and a chain of shuffles, ballots and
// reductions on each one.
//
// The trajectory is the same as the warp kernel's, decision for decision:
// step j of global phase np draws Philox {j, d, np_lo, np_hi} with the
// replica seed, target = (w0 | w1<<32) >> 1 against R' = sum_c n_c A_c, class
// = first c with target < C_c, member jj = (target - C_{c-1}) / A_c in
// row-major (= bit) order.  Domain state, edge words, counters and the open
// observation record live in global memory (L2): each visit reads its tile
// and counters, waits for its neighbours' stamped edge words, runs, and
// writes them back.  Only the domain's owner thread writes its tile,
// counters and record (and only it reads them for use: a lane without a
// domain in a round reads some domain's and discards the values), and the
// stamped edge words carry data and visit count in one 64-bit store.
//
// Scope: palindromic and fixed colour schedules, exponential and expected
// clocks, per-replica k, records at schedule endpoints or every colour pass.
// Scores, fixed-time visits and random colour orders use the warp kernel.
#pragma once

#include "kmc_kernels.cuh"

namespace kmcdev {

constexpr uint64_t TPD_COL0 = 0x0101010101010101ull; // column 0 of every row
constexpr int TPD_CACHE = 2;  // rounds of a phase whose domains a thread keeps in shared memory
constexpr int TPD_CHUNK = 32; // steps drawn at a time
constexpr int TPD_LOOK = 3;   // steps looked at in a round of events
// shared memory of a thread: 0 and the cumulative class rates, domain and
// replica of its visits, the targets of a chunk and past its end ~0 (a target
// no rate sum reaches), so that a look never reads past them
constexpr int TPD_THREAD_BYTES = 80 + 4 * TPD_CACHE * 8 + (TPD_CHUNK + TPD_LOOK) * 8;
constexpr int TPD_OBS_WORDS = 4; // open record per domain: record | steps << 32, bonds | mag << 32, mantissa, exponent

// Bit y of an 8-bit column mask to bit 8y (column 0 of row y).
__device__ __forceinline__ uint64_t tpd_col_spread(uint32_t c8)
{
    uint64_t v = ((uint64_t)(c8 & 0xFFu) * 0x0101010101010101ull) & 0x8040201008040201ull;
    return ((v + 0x7F7F7F7F7F7F7F7Full) >> 7) & TPD_COL0;
}

// Column 0 of an 8x8 tile (bits 8y) to an 8-bit mask (bit y).
__device__ __forceinline__ uint32_t tpd_col_gather(uint64_t w)
{
    return (uint32_t)(((w & TPD_COL0) * 0x0102040810204080ull) >> 56);
}

// Bit-sliced count of up neighbours (0..4) of every site of tile T, with the
// frozen halo: the N neighbour's last row hN above row 0, the S neighbour's
// first row hS below row 7, the W and E neighbours' edge columns hW, hE
// (bit y = row y) left of column 0 and right of column 7.
struct TpdPlanes {
    uint64_t b0, b1, b2;
    __device__ __forceinline__ void build(uint64_t T, uint32_t hN, uint32_t hS, uint32_t hW, uint32_t hE)
    {
        const uint64_t U = (T << 8) | (uint64_t)(hN & 0xFFu);
        const uint64_t D = (T >> 8) | ((uint64_t)(hS & 0xFFu) << 56);
        const uint64_t Wn = ((T << 1) & ~TPD_COL0) | tpd_col_spread(hW);
        const uint64_t En = ((T >> 1) & ~(TPD_COL0 << 7)) | (tpd_col_spread(hE) << 7);
        const uint64_t x = U ^ D ^ Wn, m = (U & D) | (U & Wn) | (D & Wn), k = x & En; // U + D + Wn = x + 2 m
        b0 = x ^ En;
        b1 = m ^ k;
        b2 = m & k;
    }
    // sites with exactly q up neighbours
    __device__ __forceinline__ uint64_t eq(int q) const
    {
        const uint64_t m2 = (q & 4) ? b2 : ~b2, m1 = (q & 2) ? b1 : ~b1, m0 = (q & 1) ? b0 : ~b0;
        return m2 & m1 & m0;
    }
};

// Cumulative class rates C_c = sum_{c' <= c} n_c' A_c' of tile T (classes
// 5 (s > 0) + q in order 0..9); C[9] = R'.  Of the five counts of a spin
// direction four are counted bits of the planes (q = 1 and 3 in b0, q = 2
// and 3 in b1, both in b0 b1, q = 4 in b2) and q = 0 has the rest.
// C_0 .. C_8 go to shared memory (element c + 1 of cc, element 0 holding 0;
// stride elements apart), their high words and R' stay in registers.
__device__ __forceinline__ uint64_t tpd_rates(uint64_t T, const TpdPlanes &pl, const uint64_t (&A)[10], uint32_t (&Ch)[9],
                                              uint64_t *cc, int stride)
{
    const uint32_t nup = (uint32_t)__popcll(T);
    const uint64_t b01 = pl.b0 & pl.b1;
    uint64_t acc = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const uint64_t S = s ? T : ~T;
        const uint32_t p0 = (uint32_t)__popcll(pl.b0 & S), p1 = (uint32_t)__popcll(pl.b1 & S),
                       n3 = (uint32_t)__popcll(b01 & S), n4 = (uint32_t)__popcll(pl.b2 & S);
        const uint32_t n[5] = {(s ? nup : 64u - nup) - (p0 + p1 - n3) - n4, p0 - n3, p1 - n3, n3, n4};
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            acc += (uint64_t)n[q] * A[5 * s + q];
            if (5 * s + q < 9) {
                cc[(5 * s + q + 1) * stride] = acc;
                Ch[5 * s + q < 9 ? 5 * s + q : 8] = (uint32_t)(acc >> 32);
            }
        }
    }
    return acc;
}

// Product of a normalised mantissa (value m 2^(e - 63)) and V / 2^64 where on
// (V then 2^11 or more).
__device__ __forceinline__ void tpd_mul(uint64_t &m, int &e, uint64_t V, bool on)
{
    V = on ? V : 1ull << 63;
    uint64_t hi = __umul64hi(m, V), lo = m * V;
    if ((uint32_t)(hi >> 32) == 0) { // (V below 2^33) by 32 bits first
        hi = (hi << 32) | (lo >> 32);
        lo <<= 32;
        e -= 32;
    }
    const int z = __clz((int)(uint32_t)(hi >> 32));
    const uint32_t h = __funnelshift_l((uint32_t)hi, (uint32_t)(hi >> 32), z),
                   l = __funnelshift_l((uint32_t)(lo >> 32), (uint32_t)hi, z);
    m = on ? ((uint64_t)h << 32) | l : m;
    e -= on ? z : 0;
}

// The lanes' open records go to their replicas' records (records past the
// launch's last one are dropped), as the warp kernel's flush; called by the
// whole warp, on: this lane has one to close.
template <bool EXPO>
__device__ __forceinline__ void tpd_flush(const RunParams &P, bool on, const ulonglong2 &ob, const ulonglong2 &clk, uint32_t r)
{
    const uint32_t o = (uint32_t)ob.x;
    on = on && o != NO_RECORD && (int64_t)o < P.n_obs;
    double dt = 0.0;
    if (on) dt = EXPO ? domain_time(true, clk.x, (int64_t)clk.y, 0, P.lambda) : __ddiv_rn((double)(uint32_t)(ob.x >> 32), P.lambda);
    add_to_record<false>(P, on, o, r, (int)(uint32_t)ob.y, (int)(uint32_t)(ob.y >> 32), dt, 0.0, 0.0);
}

// Persistent kernel: thread t visits, in every colour phase, the domains
// t, t + T, t + 2T, ... of that colour's list (T = threads of the grid).
// P.cta_col_off holds the five offsets of the colour-sorted domain list
// P.slot_g; P.obs_dom the open records (TPD_OBS_WORDS per domain).
//
// What bounds it: with the registers of a visit three 4-warp CTAs fit an SM,
// and three warps per scheduler issue on about half of the cycles, so a
// visit's instructions and its latency both count.  An event is some 320
// instructions and a draw 95, and one lane of 32 has an event at nearly every
// step.  So a visit first draws its steps (four at a time side by side, targets
// to shared memory), before its halo is there, and every round of events lets
// each lane look once at its own next three targets: a lane with an event takes
// it, one without sits out the round, and the warp needs about half as many
// rounds as steps.  Before that the domain's words and the halo are asked for;
// counters are added without reading them, and C_{c-1} is kept in shared
// memory.  512 uneven replicas, 60 schedules, records every 10, on 456 CTAs, at
// k = 1 / 4 / 16 / 32: 3.64 / 5.93 / 16.85 / 31.65 ms with one step per round
// and the next step's draw in line with the event, 3.77 / 5.89 / 14.37 / 26.25
// drawn first and three looked at, 3.61 / 5.59 / 14.01 / 25.71 with the halo
// asked for before the draws and no rates after a visit's last step (one 128^2
// lattice at k = 1, where every warp runs the phases in step: 13.4, 16.1, 12.9
// us a schedule).  Of drawn first: looks at two targets 5.80 / 14.79 / 27.31
// (k = 4 / 16 / 32), at four 6.03 / 14.65 / 26.64, lanes that look on until they
// find their next event no faster than one step per round; four CTAs per SM at
// 128 registers 7.72 / 18.55 / 33.68.
template <bool EXPO>
__global__ void __launch_bounds__(128, 3) tpd_kernel(const RunParams P)
{
    extern __shared__ __align__(16) uint8_t smem[];
    uint64_t *cum = reinterpret_cast<uint64_t *>(smem) + threadIdx.x; // 0, C_0 .. C_8 at stride blockDim.x
    cum[0] = 0;
    const int bd = blockDim.x;
    uint2 *cache = reinterpret_cast<uint2 *>(cum + 10 * bd); // element (colour TPD_CACHE + round) bd: {domain, replica}
    uint64_t *tg = cum + (10 + 4 * TPD_CACHE) * bd; // targets of the chunk
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int nthreads = gridDim.x * blockDim.x;
    const uint32_t *col_off = P.cta_col_off;
    const uint32_t *col_list = P.slot_g;
    const uint64_t *tile64 = reinterpret_cast<const uint64_t *>(P.tiles);
    uint64_t *tile64w = reinterpret_cast<uint64_t *>(P.tiles);
    const int nph = (P.schedule == SCHED_PALINDROME) ? 8 : 4;

    // no open record yet for any owned domain (a domain's owner is the
    // thread that visits it: list position - colour offset = tid mod T, so
    // only the owner ever reads or writes its record)
    if (P.n_obs > 0) {
        for (int c = 0; c < 4; ++c) {
            for (uint32_t i = col_off[c] + (uint32_t)tid; i < col_off[c + 1]; i += (uint32_t)nthreads) {
                uint64_t *ob = P.obs_dom + (size_t)col_list[i] * TPD_OBS_WORDS;
                ob[0] = (uint64_t)NO_RECORD;
                ob[1] = 0;
                ob[2] = 1ull << 63;
                ob[3] = 0;
            }
        }
    }

    for (int c = 0; c < 4; ++c)
        for (int m = 0; m < TPD_CACHE; ++m) {
            const uint32_t i = col_off[c] + (uint32_t)tid + (uint32_t)m * (uint32_t)nthreads;
            const uint32_t g = i < col_off[c + 1] ? col_list[i] : col_list[col_off[c]];
            cache[(c * TPD_CACHE + m) * bd] = make_uint2(g, P.dom_rep[g]);
        }
    unsigned spins = 0; // halo re-reads (profiling)
    bool ok = true;
    uint32_t gc0 = 0, gc1 = 0, gc2 = 0, gc3 = 0; // completed visit groups per colour in this launch
    const uint64_t gp_begin = (uint64_t)P.sched_begin * nph;
    const uint64_t gp_end = (uint64_t)(P.sched_begin + P.n_sched) * nph;
    uint64_t gp = gp_begin;
    while (gp < gp_end) {
        const uint64_t n = gp / nph;
        const int p = (int)(gp % nph);
        const uint64_t np0 = n * 8 + (uint64_t)p;
        const int colour = fixed_colour(P.schedule, p);
        // fuse following phases of the same colour unless an observation intervenes
        int nf = 1;
        while (!P.obs_pass && gp + nf < gp_end) {
            const uint64_t g2 = gp + nf;
            const int p2 = (int)(g2 % nph);
            if (fixed_colour(P.schedule, p2) != colour) break;
            if (p2 == 0) {
                const int64_t nl_prev = (int64_t)(g2 / nph - 1 - (uint64_t)P.sched_begin);
                if (P.obs_every > 0 && ((nl_prev + 1) % P.obs_every) == 0) break;
            }
            ++nf;
        }
        auto gcount = [&](int c) { return c == 0 ? gc0 : c == 1 ? gc1 : c == 2 ? gc2 : gc3; };
        // a neighbour across a row has colour ^ 2, across a column colour ^ 1
        const uint32_t needNS = gcount(colour ^ 2) + (uint32_t)P.debug_extra;
        const uint32_t needWE = gcount(colour ^ 1) + (uint32_t)P.debug_extra;
        const uint32_t after = gcount(colour) + 1;
        const int64_t pass = (int64_t)(gp - gp_begin);
        // Rounds of one domain per thread: every lane of a warp runs the
        // same trip counts (lanes without a domain in a round ride along
        // predicated), so the halo wait and the steps stay warp-synchronous
        // and the collectives below see the full warp.
        const uint32_t lo = col_off[colour], hi = col_off[colour + 1];
        const uint32_t rounds = (hi - lo + (uint32_t)nthreads - 1) / (uint32_t)nthreads;
        for (uint32_t m = 0; m < rounds && ok; ++m) {
            const uint32_t i = lo + (uint32_t)tid + m * (uint32_t)nthreads;
            const bool has = i < hi;
            uint2 gr;
            if (m < TPD_CACHE) {
                gr = cache[(colour * TPD_CACHE + (int)m) * bd];
            } else {
                gr.x = has ? col_list[i] : col_list[lo];
                gr.y = P.dom_rep[gr.x];
            }
            const uint32_t g = gr.x, r = gr.y;
            const uint32_t base = __ldg(&P.rep_dom_off[r]);
            const uint32_t Dx = (uint32_t)__ldg(&P.rep_Dx[r]);
            const int k = __ldg(&P.rep_k[r]);
            const uint64_t seed = __ldg(&P.rep_seed[r]);
            uint64_t A[10];
#pragma unroll
            for (int c = 0; c < 10; ++c) A[c] = __ldg(&P.rep_A[(size_t)r * RATE_WORDS + c]);
            const uint32_t d = g - base;
            const uint32_t by = d / Dx, bx = d - by * Dx;
            const uint32_t gN = by == 0 ? g + (Dx - 1) * Dx : g - Dx, gS = by == Dx - 1 ? g - (Dx - 1) * Dx : g + Dx;
            const uint32_t gW = bx == 0 ? g + Dx - 1 : g - 1, gE = bx == Dx - 1 ? g - (Dx - 1) : g + 1;
            const int total = has ? nf * k : 0;
            const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
            uint64_t vM = 1ull << 63;
            int vE = 0;
            const int smax = (int)__reduce_max_sync(FULL_WARP, (unsigned)total);
            // Step st = f k + j of the visit is step j of global phase np0 + f: its
            // target (~0 past the last step), and its clock variate into the
            // visit's product.
            auto draw = [&](int st) {
                const bool act = st < total;
                const int f = st >= k ? 1 : 0; // at most two phases fuse
                const uint64_t np = np0 + (uint64_t)f;
                const uint4 w = philox4x32_10(make_uint4((uint32_t)(st - (f ? k : 0)), d, (uint32_t)np,
                                                         (uint32_t)(np >> 32) & 0xFFFFFFu), key);
                if (EXPO) {
                    // clock variate v = V 2^-53, V the top 53 bits plus 1 (2^53 wraps
                    // to 0: v = 1 leaves the product)
                    const uint64_t V = ((((uint64_t)w.w << 32) | w.z) & ~0x7FFull) + 0x800ull;
                    tpd_mul(vM, vE, V, act && V != 0);
                }
                return act ? (((uint64_t)w.y << 32) | w.x) >> 1 : ~0ull;
            };
            // the targets of steps base .. base + 31 of the visit to shared memory
            auto draw_chunk = [&](int base) {
                const int n = min(TPD_CHUNK, smax - base);
#pragma unroll 1
                for (int i = 0; i + 4 <= n; i += 4) {
                    uint64_t t[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) t[u] = draw(base + i + u);
#pragma unroll
                    for (int u = 0; u < 4; ++u) tg[(i + u) * bd] = t[u];
                }
#pragma unroll 1
                for (int i = n & ~3; i < n; ++i) tg[i * bd] = draw(base + i);
#pragma unroll
                for (int u = 0; u < TPD_LOOK; ++u) tg[(n + u) * bd] = ~0ull;
            };
            // The domain's words and the halo are asked for before the draws, which
            // take longer than they do, but after everything above: asked for
            // first, the domain's words took the addresses' loads with them
            // (1300 cycles instead of 520 up to the first read of the halo).
            uint64_t T = tile64[g];
            uint64_t *ctr = P.dctr + (size_t)g * DCTR_WORDS;
            uint64_t H = ctr[DCTR_HASH];
            uint64_t clkM = ctr[DCTR_CLKM];
            int64_t clkE = (int64_t)ctr[DCTR_CLKE];
            const int64_t o = P.n_obs > 0 ? (P.obs_pass ? pass : pass / nph) / P.obs_every : 0;
            uint64_t *ob = P.obs_dom + (size_t)g * TPD_OBS_WORDS;
            ulonglong2 ob01 = make_ulonglong2(0, 0), obM = make_ulonglong2(0, 0);
            if (P.n_obs > 0) {
                ob01 = *reinterpret_cast<const ulonglong2 *>(ob);
                obM = *reinterpret_cast<const ulonglong2 *>(ob + 2);
            }
            // Halo: the N neighbour's S row, the S neighbour's N row, the W
            // neighbour's E column, the E neighbour's W column (half 0 of
            // each), stamped with the neighbour's completed visits; looked at
            // after the draws, when the warp re-reads until every lane's four
            // are current (bounded)
            const uint64_t *pN = P.edges + (size_t)gN * EDGE_WORDS + 2 * EDGE_S;
            const uint64_t *pS = P.edges + (size_t)gS * EDGE_WORDS + 2 * EDGE_N;
            const uint64_t *pW = P.edges + (size_t)gW * EDGE_WORDS + 2 * EDGE_E;
            const uint64_t *pE = P.edges + (size_t)gE * EDGE_WORDS + 2 * EDGE_W;
            uint64_t wN = 0, wS = 0, wW = 0, wE = 0;
            auto current = [&]() {
                return !has || ((uint32_t)(wN >> 32) >= needNS && (uint32_t)(wS >> 32) >= needNS &&
                                (uint32_t)(wW >> 32) >= needWE && (uint32_t)(wE >> 32) >= needWE);
            };
            if (has) {
                wN = ld_volatile_global(pN);
                wS = ld_volatile_global(pS);
                wW = ld_volatile_global(pW);
                wE = ld_volatile_global(pE);
            }
            draw_chunk(0);
            bool ready = current();
            if (!__all_sync(FULL_WARP, ready)) {
                const uint64_t t0 = global_ns();
                unsigned n = 0;
                while (true) {
                    if (!ready) {
                        wN = ld_volatile_global(pN);
                        wS = ld_volatile_global(pS);
                        wW = ld_volatile_global(pW);
                        wE = ld_volatile_global(pE);
                        ++spins;
                        ready = current();
                    }
                    if (__all_sync(FULL_WARP, ready)) break;
                    if ((++n & 63u) == 0) {
                        const bool late = global_ns() - t0 > P.bar_limit_ns;
                        const bool quit = late || *(volatile int *)P.err != 0;
                        if (__any_sync(FULL_WARP, quit)) {
                            if (late) atomicCAS(P.err, 0, ERR_TIMEOUT);
                            ok = false;
                            break;
                        }
                    }
                }
                if (!ok) break;
            }
            const uint32_t hN = (uint32_t)wN, hS = (uint32_t)wS, hW = (uint32_t)wW, hE = (uint32_t)wE;

            TpdPlanes pl;
            pl.build(T, hN, hS, hW, hE);
            uint32_t Ch[9];
            uint64_t R = tpd_rates(T, pl, A, Ch, cum, bd);
            uint32_t flips = 0;
            int dbonds = 0, dmag = 0;
            for (int base = 0; base < smax; base += TPD_CHUNK) {
                if (base > 0) draw_chunk(base);
                const int n = min(TPD_CHUNK, smax - base);
                int pos = 0; // this lane's next step of the chunk
                for (bool go = true; go;) {
                    // the first of the next steps that is no null step (App. A: the
                    // diagonal 1 - R/n_d), else the last of them
                    uint64_t t[TPD_LOOK];
#pragma unroll
                    for (int u = 0; u < TPD_LOOK; ++u) t[u] = tg[(pos + u) * bd];
                    uint64_t tgt = t[TPD_LOOK - 1];
                    int off = TPD_LOOK - 1;
#pragma unroll
                    for (int u = TPD_LOOK - 2; u >= 0; --u) {
                        const bool e = t[u] < R;
                        tgt = e ? t[u] : tgt;
                        off = e ? u : off;
                    }
                    const bool ev = tgt < R;
                    const int st = base + pos + off;
                    pos = min(pos + off + 1, n);
                    go = __any_sync(FULL_WARP, pos < n);
                    // a lane without an event runs the event with no effect
                    if (!__any_sync(FULL_WARP, ev)) continue;
                    // class: the first c with tgt < C_c; by the high words it may come
                    // out too high where those are equal
                    int c = 0;
                    const uint32_t th = (uint32_t)(tgt >> 32);
#pragma unroll
                    for (int cc = 0; cc < 9; ++cc) c += (th >= Ch[cc]) ? 1 : 0;
                    uint64_t Cprev = cum[c * bd];
                    while (tgt < Cprev) Cprev = cum[--c * bd];
                    const uint64_t Ac = __ldg(&P.rep_A[(size_t)r * RATE_WORDS + c]);
                    // exact jj = floor((tgt - C_{c-1}) / A_c) < n_c <= 64: an FP32
                    // estimate rounded toward the lower side is jj or jj - 1, and
                    // one integer comparison decides which
                    const uint64_t x = tgt - Cprev;
                    const float inv = __frcp_rd(u64_to_float_ru(Ac));
                    uint32_t jj = (uint32_t)__fmul_rz(u64_to_float_rz(x), inv);
                    jj = (x - (uint64_t)jj * Ac >= Ac) ? jj + 1u : jj;
                    const int qc = (c >= 5) ? c - 5 : c;
                    const uint64_t mask = ((c >= 5) ? T : ~T) & pl.eq(qc);
                    const int site = select_bit(mask, jj) & 63;
                    T ^= ev ? 1ull << site : 0ull;
                    const int f = st >= k ? 1 : 0;
                    const uint64_t np = np0 + (uint64_t)f;
                    const uint64_t h = (H ^ ((np << 32) | ((uint64_t)(st - (f ? k : 0)) << 16) | (uint64_t)site)) * HASH_PRIME;
                    H = ev ? h : H;
                    flips += ev ? 1u : 0u;
                    // flipping spin s with neighbour sum 2 qc - 4 changes the bond
                    // sum by -2 s (2 qc - 4) and the magnetisation by -2 s
                    const int g2 = ev ? (c >= 5 ? -2 : 2) : 0;
                    dbonds += g2 * (2 * qc - 4);
                    dmag += g2;
                    if (go || base + n < smax) { // (else the visit is over)
                        pl.build(T, hN, hS, hW, hE);
                        R = tpd_rates(T, pl, A, Ch, cum, bd);
                    }
                }
            }
            // edges first (neighbours wait for them), then tile, counters and record
            if (has) {
                uint64_t *ew = P.edges + (size_t)g * EDGE_WORDS;
                const uint64_t cnt = (uint64_t)after << 32;
                st_cg(ew + 2 * EDGE_N, cnt | (T & 0xFFull));
                st_cg(ew + 2 * EDGE_S, cnt | (T >> 56));
                st_cg(ew + 2 * EDGE_W, cnt | tpd_col_gather(T));
                st_cg(ew + 2 * EDGE_E, cnt | tpd_col_gather(T >> 7));
            }
            // the visit's changes belong to the first record at or after its pass
            const bool turn = P.n_obs > 0 && has && (int64_t)(uint32_t)ob01.x != o;
            if (__any_sync(FULL_WARP, turn)) tpd_flush<EXPO>(P, turn, ob01, obM, r);
            if (!has) continue;
            if (EXPO) mant_mul(clkM, clkE, vM, (int64_t)vE); // the domain clock takes the visit's product
            if (flips) {
                tile64w[g] = T;
                ctr[DCTR_HASH] = H;
                atomicAdd(reinterpret_cast<unsigned long long *>(ctr + DCTR_FLIPS), (unsigned long long)flips);
            }
            atomicAdd(reinterpret_cast<unsigned long long *>(ctr + DCTR_STEPS), (unsigned long long)total); // (no result: no wait)
            if (EXPO) {
                ctr[DCTR_CLKM] = clkM;
                ctr[DCTR_CLKE] = (uint64_t)clkE;
            }
            if (P.n_obs > 0) {
                uint64_t om = obM.x;
                int64_t oe = (int64_t)obM.y;
                if ((int64_t)(uint32_t)ob01.x != o) {
                    ob01 = make_ulonglong2((uint64_t)(uint32_t)o, 0);
                    om = 1ull << 63;
                    oe = 0;
                }
                const uint32_t steps = (uint32_t)(ob01.x >> 32) + (uint32_t)total;
                const int bonds = (int)(uint32_t)ob01.y + dbonds, mag = (int)(uint32_t)(ob01.y >> 32) + dmag;
                if (EXPO) mant_mul(om, oe, vM, (int64_t)vE);
                *reinterpret_cast<ulonglong2 *>(ob) = make_ulonglong2(
                    (uint64_t)(uint32_t)o | ((uint64_t)steps << 32), (uint64_t)(uint32_t)bonds | ((uint64_t)(uint32_t)mag << 32));
                *reinterpret_cast<ulonglong2 *>(ob + 2) = make_ulonglong2(om, (uint64_t)oe);
            }
        }
        if (colour == 0) ++gc0;
        else if (colour == 1) ++gc1;
        else if (colour == 2) ++gc2;
        else ++gc3;
        gp += (uint64_t)nf;
    }
    if (P.polls && spins != 0) atomicAdd(P.polls, (unsigned long long)spins);
    if (__any_sync(FULL_WARP, !ok || *(volatile int *)P.err != 0)) return; // (whole warps: records are closed by the warp)
    // every owned domain's open record
    if (P.n_obs > 0) {
        for (int c = 0; c < 4; ++c) {
            const uint32_t lo = col_off[c], hi = col_off[c + 1];
            const uint32_t rounds = (hi - lo + (uint32_t)nthreads - 1) / (uint32_t)nthreads;
            for (uint32_t m = 0; m < rounds; ++m) {
                const uint32_t i = lo + (uint32_t)tid + m * (uint32_t)nthreads;
                const uint32_t g = i < hi ? col_list[i] : col_list[lo];
                const ulonglong2 *ob = reinterpret_cast<const ulonglong2 *>(P.obs_dom + (size_t)g * TPD_OBS_WORDS);
                tpd_flush<EXPO>(P, i < hi, ob[0], ob[1], P.dom_rep[g]);
            }
        }
    }
}

} // namespace kmcdev
