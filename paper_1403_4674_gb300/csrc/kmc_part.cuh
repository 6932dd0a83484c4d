// kmc_part.cuh -- sm_103a device code for small periodic lattices (L <= 128)
// under the partitions of Sec. 3.2: a Dx x Dx grid of square blocks or N_D
// vertical stripes of width L/N_D and full height (Fig. 1 caption), with any
// domain size n_d (the paper's 12^2 and 100^2 lattices).
//
// Data parallelism is over trajectories (the paper's N_TRAJ runs per
// setting): one warp owns one trajectory for the whole launch and runs its
// domain processes in schedule order, so the halo of a visit is the live
// state -- no other domain of the trajectory moves meanwhile.  The lattice
// lives in shared memory as bit rows (PART_ROW32 words each), beside the
// class counts of every domain and, where they fit, of every domain row; a
// flip updates the counts of the five sites it touches, whichever domains
// they lie in, so a visit starts from its counts without a recount.
//
// What bounds it is one warp's chain of real events (the paper's 50
// trajectories leave two SMs of three idle, and a trajectory has no work for
// a second warp): ncu counts 1.0 warps per scheduler that has any, issue
// 24 % of its cycles, the stalls led by fixed-latency dependencies.  So the
// steps of a trajectory are drawn 32 at a time across visits and schedules
// (a window: one lane per step, whole visits of up to 32 steps each or 32
// steps of a longer one), null runs cost nothing (the next event of the
// window is one vote away), and the event's chain is kept short: the class
// from the cumulative rates in every lane alike, the member's row from
// 16 domain rows per lane of the rows' counts, its column from a
// lane-parallel bit count, the five sites' classes from five lanes side by
// side, the counts by shared-memory atomics.  Measured one visit after the
// other, with the windows and now: 50 trajectories of 100^2 in four stripes,
// k = 5, random order, 800 schedules 3.22, 1.89, 1.20 ms; 500 of 12^2 in four
// blocks, k = 1, 4000 schedules 11.1, 5.81, 3.11 ms.  Section clocks of one
// trajectory of each, cycles: an event 1630 and 1500 (of it about: rates 240,
// class 245, row 190-320, column 268, neighbours 143, counts 295), a window
// 1030 and 2120 (its orders and draws 730 and 1350, the last look that finds
// no event 240, records 70 and 520), staging and writing back 130,000 and
// 21,000 once.  16,000 steps are 500 windows with about 1000 events (one step
// in 16, the stripes) or 2400 (one in 6.6, the blocks), so events are 0.8 of
// 1.2 ms and 1.8 of 3.1 ms.
//
// Step target (n_d not a power of two): P = 63 - ceil(log2 n_d),
// M = n_d 2^P, target = floor(X M / 2^64) for X = w0 | w1<<32; with n_d a
// power of two this is X >> 1, the lattice path's target.
#pragma once

#include <cstdint>

#include "kmc_kernels.cuh"

namespace kmcpart {

using kmcdev::FULL_WARP;
using kmcdev::HASH_PRIME;
using u128 = unsigned __int128;

constexpr int PART_WARPS = 1;        // trajectories per CTA: few trajectories spread over the SMs
constexpr int PART_MAX_L = 128;
constexpr int PART_PHASE_SLOTS = 64; // Philox phase index np = n*64 + p
constexpr int PART_BLOCKS = 0, PART_STRIPES = 1;
constexpr uint32_t PART_TAG_PERM = 2u;
// Bit rows in shared memory: PART_ROW32 32-bit words per row, bit x + 1 =
// column x (1 = up), bit 0 a copy of column L - 1 and bit L + 1 one of column
// 0, so that a window of columns and their W and E neighbours is a shift.
constexpr int PART_ROW32 = 6;
// The class counts of domain rows are kept (u8 [N_D][10][rows], the rows
// padded to a multiple of 16: one 128-bit load each 16 rows) when the
// lattice has at most PART_RC_ROWS padded domain rows.  Otherwise an event
// counts its domain's rows, four a lane over the whole warp (16 a lane on the
// few lanes that would load them took 2.4 times as long: 1000 trajectories of
// 100^2 in ten stripes, k = 5, 79 and 32 us a schedule).
constexpr int PART_RC_ROWS = 1024;
constexpr int PART_ORDER_BYTES = 1024;
// shared memory of a trajectory in bytes: the class counts of the domain
// rows, the fixed-point rates and their reciprocals (u64 [10][2]), the class
// counts of every domain (u32 [N_D][12], ten used), the bit rows, the domains
// of the visits (u8: the random orders of the schedules in use, or one colour
// schedule's visits and after them their phases), each domain's neighbours
// (u8 [N_D][4]) and its first column and row (u8 [N_D][2])
struct PartLayout {
    int rc, atab, dcount, rows, order, nbd, org, bytes;
    __host__ __device__ PartLayout(int L, int ND, int Hd)
    {
        const int Hp = (Hd + 15) & ~15;
        rc = 0;
        atab = (ND * Hp <= PART_RC_ROWS) ? ND * Hp * 10 : 0;
        dcount = atab + 160;
        rows = dcount + ND * 48;
        order = rows + L * PART_ROW32 * 4;
        nbd = order + PART_ORDER_BYTES;
        org = nbd + ND * 4;
        bytes = (org + ND * 2 + 15) & ~15;
    }
};

struct PartParams {
    int n_traj, L, kind, ND, k;
    int Dx;              // blocks per side (blocks), else 0
    int W, H;            // domain width and height
    int ncol;            // colours (1, 2 or 4)
    int schedule, obs_every;
    int64_t sched_begin, n_sched;
    uint64_t M;          // n_d 2^P
    double J, nu;
    const uint64_t *seed; // [n_traj]
    const uint64_t *A;    // [n_traj][10]
    const double *h;      // [n_traj]
    int8_t *spins;        // [n_traj][L][L], +-1
    uint64_t *hash, *clkM;
    int64_t *clkE, *flips, *steps;
    double *t;            // [n_traj] clock after the launch
    double *obs;          // [n_rec][n_traj][4] or null
    int *err;
};

// Row y, bit x = column x.
__device__ __forceinline__ u128 row_ld(const uint32_t *rows, int y, u128 Lm)
{
    const uint32_t *w = rows + PART_ROW32 * y;
    const uint64_t lo = ((uint64_t)w[1] << 32) | w[0], hi = ((uint64_t)w[3] << 32) | w[2];
    return ((((u128)hi << 64 | lo) >> 1) | ((u128)w[4] << 127)) & Lm;
}

// bit x <- bit x-1 (mod L) / bit x <- bit x+1 (mod L) of an L-bit row
__device__ __forceinline__ u128 rot_w(u128 c, int L, u128 Lm) { return ((c << 1) | (c >> (L - 1))) & Lm; }
__device__ __forceinline__ u128 rot_e(u128 c, int L) { return (c >> 1) | ((c & (u128)1) << (L - 1)); }

__device__ __forceinline__ int popc128(u128 v) { return __popcll((uint64_t)v) + __popcll((uint64_t)(v >> 64)); }

// Up-neighbour count planes (bit-sliced b2 b1 b0) of row y, restricted to the
// domain columns DM, and its up / down spins there.
struct RowPlanes {
    u128 up, dn, b0, b1, b2;
};

__device__ __forceinline__ RowPlanes row_planes(const uint32_t *rows, int y, int L, u128 Lm, u128 DM)
{
    const u128 c = row_ld(rows, y, Lm);
    const u128 n = row_ld(rows, (y == 0) ? L - 1 : y - 1, Lm);
    const u128 s = row_ld(rows, (y == L - 1) ? 0 : y + 1, Lm);
    const u128 w = rot_w(c, L, Lm), e = rot_e(c, L);
    const u128 s1 = n ^ s, c1 = n & s, s2 = w ^ e, c2 = w & e, t0 = s1 & s2;
    RowPlanes p;
    p.b0 = s1 ^ s2;
    p.b1 = c1 ^ c2 ^ t0;
    p.b2 = (c1 & c2) | (c1 & t0) | (c2 & t0);
    p.up = c & DM;
    p.dn = ~c & DM;
    return p;
}

// Sites of class c = 5 up + q in a row.
__device__ __forceinline__ u128 class_mask(const RowPlanes &p, int c)
{
    const int q = (c >= 5) ? c - 5 : c;
    const u128 ones = ~(u128)0;
    const u128 diff = (p.b2 ^ ((q & 4) ? ones : 0)) | (p.b1 ^ ((q & 2) ? ones : 0)) | (p.b0 ^ ((q & 1) ? ones : 0));
    return ((c >= 5) ? p.up : p.dn) & ~diff;
}

// Lane c (< 10) receives n_c of the domain (rows y0 .. y0+H-1).
__device__ __forceinline__ uint32_t part_counts(const uint32_t *rows, int lane, int y0, int H, int RPL, int L,
                                                u128 Lm, u128 DM)
{
    uint32_t w[5] = {0, 0, 0, 0, 0};
    for (int t = 0; t < RPL; ++t) {
        const int yy = lane * RPL + t;
        if (yy >= H) break;
        const RowPlanes p = row_planes(rows, y0 + yy, L, Lm, DM);
        const u128 n2 = ~p.b2;
        const u128 e[5] = {n2 & ~p.b1 & ~p.b0, n2 & ~p.b1 & p.b0, n2 & p.b1 & ~p.b0, n2 & p.b1 & p.b0, p.b2};
#pragma unroll
        for (int q = 0; q < 5; ++q)
            w[q] += (uint32_t)popc128(p.dn & e[q]) | ((uint32_t)popc128(p.up & e[q]) << 16);
    }
    uint32_t tw = 0;
    const int q = (lane < 5) ? lane : lane - 5;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const uint32_t s = __reduce_add_sync(FULL_WARP, w[i]);
        if (q == i) tw = s;
    }
    const uint32_t n = (lane < 5) ? (tw & 0xFFFFu) : (tw >> 16);
    return (lane < 10) ? n : 0u;
}

// Class 5 up + (number of up neighbours) of site (x, y), from the live rows.
__device__ __forceinline__ int site_class(const uint32_t *rows, int x, int y, int ym, int yp)
{
    auto bit = [&](int b, int yy) { return (int)((rows[PART_ROW32 * yy + (b >> 5)] >> (b & 31)) & 1u); };
    return 5 * bit(x + 1, y) + bit(x, y) + bit(x + 2, y) + bit(x + 1, ym) + bit(x + 1, yp);
}

// One warp runs one trajectory's steps in windows of 32 consecutive steps of
// its sequence (schedule after schedule, visit after visit), whatever visits
// they belong to: lane i draws step i of the window and holds its domain,
// its target and that domain's cumulative class rates.  A null step changes
// nothing, so one ballot of target < R' over the lanes finds the next real
// event of the whole window, in whichever visit it falls; every lane has
// formed its own step's class and member index by then, and after the event
// each lane forms its domain's rates again from the class counts in shared
// memory.  What a trajectory costs is thus one chain per real event (at T =
// 2.4 one step in 6 to 16) and a fixed part per 32 steps, where a loop
// over visits paid a fixed part per visit.  Records between the window's
// steps come from per-lane copies of the bond sum and the magnetisation and
// from the inclusive products of the clock variates; the lanes at whose
// steps a pass with a record ends write them side by side.
template <bool EXPO>
__global__ void __launch_bounds__(PART_WARPS * 32) part_kernel(const PartParams P)
{
    extern __shared__ __align__(16) uint8_t part_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tr = blockIdx.x * PART_WARPS + warp;
    if (tr >= P.n_traj) return; // whole warps only; no CTA-wide barrier below
    const int L = P.L, ND = P.ND;
    const PartLayout lay(L, ND, P.H);
    uint8_t *base8 = part_smem + (size_t)warp * lay.bytes;
    uint32_t *rows = reinterpret_cast<uint32_t *>(base8 + lay.rows);
    uint8_t *order = base8 + lay.order;
    uint8_t *nbd = base8 + lay.nbd;                                     // [N_D][4] W, E, N, S domains
    uint8_t *org = base8 + lay.org;                                     // [N_D][2] first column and row
    uint32_t *dcount = reinterpret_cast<uint32_t *>(base8 + lay.dcount); // [N_D][12] class counts
    ulonglong2 *atab = reinterpret_cast<ulonglong2 *>(base8 + lay.atab); // [10] A_c, floor((2^64 - 1) / A_c)
    uint8_t *rc = base8 + lay.rc;                                       // [N_D][10][Hp]
    const u128 Lm = (L == 128) ? ~(u128)0 : (((u128)1 << L) - 1);
    const int8_t *sp = P.spins + (size_t)tr * L * L;

    // load the lattice into bit rows (ballots over 32-column chunks)
    int bad = 0;
    for (int y = 0; y < L; ++y) {
        // bit b: column b - 1, with wrap
        for (int b0 = 0; b0 < 32 * PART_ROW32; b0 += 32) {
            const int b = b0 + lane;
            const int x = (b == 0) ? L - 1 : (b == L + 1) ? 0 : b - 1;
            const int8_t v = (b < L + 2) ? sp[(size_t)y * L + x] : (int8_t)-1;
            bad |= (v != 1 && v != -1);
            const uint32_t w = __ballot_sync(FULL_WARP, v == 1);
            if (lane == 0) rows[PART_ROW32 * y + (b0 >> 5)] = w;
        }
    }
    if (__any_sync(FULL_WARP, bad) && lane == 0) atomicOr(P.err, 1);
    __syncwarp();

    uint64_t A[10];
#pragma unroll
    for (int c = 0; c < 10; ++c) A[c] = P.A[(size_t)tr * 10 + c];
    const uint64_t seed = P.seed[tr];
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    const double hr = P.h[tr];
    uint64_t H = P.hash[tr], clkM = P.clkM[tr];
    int64_t clkE = P.clkE[tr], flips = P.flips[tr];
    const int64_t steps0 = P.steps[tr];
    const int W = P.W, Hd = P.H, k = P.k;
    const int Hp = (Hd + 15) & ~15;
    const u128 DM0 = (W == 128) ? ~(u128)0 : (((u128)1 << W) - 1);
    const uint64_t M = P.M;
    const bool stripes = P.kind == PART_STRIPES;
    const int nbx = stripes ? ND : P.Dx, nby = stripes ? 1 : P.Dx; // domains per row and column

    const bool use_rc = ND * Hp <= PART_RC_ROWS;
    const int rpl = use_rc ? 16 : 4; // rows per lane in an event
    if (lane < 10) {
        const uint64_t Al = P.A[(size_t)tr * 10 + lane];
        atab[lane] = make_ulonglong2(Al, Al ? ~0ull / Al : 0ull);
    }
    for (int d = lane; d < ND; d += 32) {
        const int bx = d % nbx, by = d / nbx;
        org[2 * d] = (uint8_t)(bx * W);
        org[2 * d + 1] = (uint8_t)(by * Hd);
        nbd[4 * d + 0] = (uint8_t)(by * nbx + (bx == 0 ? nbx - 1 : bx - 1));
        nbd[4 * d + 1] = (uint8_t)(by * nbx + (bx == nbx - 1 ? 0 : bx + 1));
        nbd[4 * d + 2] = (uint8_t)((by == 0 ? nby - 1 : by - 1) * nbx + bx);
        nbd[4 * d + 3] = (uint8_t)((by == nby - 1 ? 0 : by + 1) * nbx + bx);
    }
    // class counts of every domain (and of every domain row, when they
    // fit), kept up to date flip by flip
    for (int d = 0; d < ND; ++d) {
        const int x0 = (d % nbx) * W, y0 = (d / nbx) * Hd;
        const uint32_t n = part_counts(rows, lane, y0, Hd, (Hd + 31) / 32, L, Lm, DM0 << x0);
        if (lane < 12) dcount[d * 12 + lane] = n;
        if (use_rc) {
            for (int yy = lane; yy < Hp; yy += 32) {
                const RowPlanes pr = row_planes(rows, y0 + min(yy, Hd - 1), L, Lm, DM0 << x0);
                for (int c = 0; c < 10; ++c)
                    rc[(d * 10 + c) * Hp + yy] = (yy < Hd) ? (uint8_t)popc128(class_mask(pr, c)) : (uint8_t)0;
            }
        }
    }

    const bool perm = P.schedule == kmcdev::SCHED_RANDOM_PERM;
    const int nph = perm ? ND : (P.schedule == kmcdev::SCHED_PALINDROME ? 2 * P.ncol : P.ncol);
    const int dpp = (perm || ND == 1) ? 1 : ND / P.ncol; // visits per phase
    const int Vs = nph * dpp;                             // visits per schedule
    const double N = (double)L * (double)L;
    uint8_t *phase_of = order + 128; // colour schedules: the phase of visit v (Vs <= 128)
    if (!perm) {
        // colour of phase p: 0 1 .. [.. 1 0]; the i-th domain of colour col in
        // ascending order (blocks: by = col>>1 + 2 (i / (Dx/2)), bx = col&1 + 2 (i % (Dx/2)))
        for (int v = lane; v < Vs; v += 32) {
            const int p = v / dpp, i = v - p * dpp;
            const int col = (p < P.ncol) ? p : (2 * P.ncol - 1 - p);
            int d = 0;
            if (ND > 1) {
                const int half = P.Dx / 2;
                d = stripes ? col + 2 * i : ((col >> 1) + 2 * (i / half)) * P.Dx + (col & 1) + 2 * (i % half);
            }
            order[v] = (uint8_t)d;
            phase_of[v] = (uint8_t)p;
        }
    }
    __syncwarp();

    // bond sum = 2 L^2 - 2 (unlike neighbour pairs), magnetisation = 2 (up spins) - L^2
    const bool want = P.obs != nullptr && P.obs_every > 0;
    int bonds = 0, mag = 0;
    if (want) {
        int unlike = 0, up = 0;
        for (int y = lane; y < L; y += 32) {
            const u128 c = row_ld(rows, y, Lm);
            const u128 s = row_ld(rows, (y == L - 1) ? 0 : y + 1, Lm);
            unlike += popc128((c ^ rot_e(c, L)) & Lm) + popc128(c ^ s);
            up += popc128(c);
        }
        bonds = 2 * L * L - 2 * __reduce_add_sync(FULL_WARP, unlike);
        mag = 2 * __reduce_add_sync(FULL_WARP, up) - L * L;
    }
    auto write_record = [&](int64_t rec, int b, int mg, uint64_t cm, int64_t ce, int64_t st) {
        const double e = __ddiv_rn(__dsub_rn(__dmul_rn(-P.J, (double)b), __dmul_rn(hr, (double)mg)), N);
        const double m = __ddiv_rn((double)mg, N);
        double4_32a v;
        v.x = e;
        v.y = m;
        v.z = __dmul_rn(e, m);
        v.w = kmcdev::domain_time(EXPO, cm, ce, st, __dmul_rn(N, P.nu));
        reinterpret_cast<double4_32a *>(P.obs)[(size_t)rec * P.n_traj + tr] = v;
    };

    // The paper's random order of all domains of a schedule (Fisher-Yates over
    // Philox), one schedule per lane, into a ring of n_ord schedules.
    int n_ord = 64;
    while (n_ord * ND > PART_ORDER_BYTES) n_ord >>= 1; // a power of two, >= 16
    int64_t ord_end = 0; // schedules shuffled so far
    auto shuffle = [&](int64_t nl) {
        uint8_t *ord = order + (int)(nl & (n_ord - 1)) * ND;
        const uint64_t n = (uint64_t)(P.sched_begin + nl);
        for (int i = 0; i < ND; ++i) ord[i] = (uint8_t)i;
        for (int i = ND - 1; i >= 1; --i) {
            const uint4 w = kmcdev::philox4x32_10(
                make_uint4((uint32_t)i, 0u, (uint32_t)n, ((uint32_t)(n >> 32) & 0xFFFFFFu) | (PART_TAG_PERM << 24)),
                key);
            const int jx = (int)__umul64hi(((uint64_t)w.y << 32) | w.x, (uint64_t)(i + 1));
            const uint8_t tmp = ord[i];
            ord[i] = ord[jx];
            ord[jx] = tmp;
        }
    };

    // The clock: each lane multiplies the variates of its own steps, and the
    // lanes' products are combined only where a record or the launch's end
    // asks for them.  A step takes 1.44 off the exponent on average: past
    // 1.49e9 steps of a trajectory the joined exponent leaves 32 bits.
    uint64_t lM = 1ull << 63;
    int64_t lE = 0;
    auto join = [&]() {
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint64_t m2 = __shfl_xor_sync(FULL_WARP, lM, off);
            const int64_t e2 = __shfl_xor_sync(FULL_WARP, (long long)lE, off);
            kmcdev::mant_mul(lM, lE, m2, e2);
        }
        kmcdev::mant_mul(clkM, clkE, __shfl_sync(FULL_WARP, lM, 0), (int64_t)__shfl_sync(FULL_WARP, (long long)lE, 0));
        lM = 1ull << 63;
        lE = 0;
    };
    // neighbour of this lane (lanes 1..4: W, E, N, S; lane 0: the site)
    const int dxl = (lane == 1) ? -1 : (lane == 2) ? 1 : 0, dyl = (lane == 3) ? -1 : (lane == 4) ? 1 : 0;

    const int64_t total = P.n_sched * (int64_t)Vs * k;
    // this lane's step: schedule nl (of this launch), visit v, step j of it;
    // 32 steps on are 32 / k visits and 32 % k steps on
    int64_t nl = 0;
    int v = 0, j = 0;
    if (k > 0) {
        const int q = lane / k;
        j = lane - q * k;
        nl = q / Vs;
        v = q - (int)nl * Vs;
    }
    const int jump_j = k > 0 ? 32 % k : 0, jump_v = k > 0 ? (32 / k) % Vs : 0, jump_n = k > 0 ? (32 / k) / Vs : 0;
    for (int64_t s0 = 0; s0 < total; s0 += 32) {
        const bool act = s0 + lane < total;
        if (perm) {
            // a window spans at most n_ord / 2 schedules, so the half of the
            // ring that is filled here holds none of its orders
            const int64_t last = __shfl_sync(FULL_WARP, (long long)nl, 31);
            while (ord_end <= last && ord_end < P.n_sched) {
                __syncwarp();
                if (lane < n_ord / 2 && ord_end + lane < P.n_sched) shuffle(ord_end + lane);
                ord_end += n_ord / 2;
                __syncwarp();
            }
        }
        int d = 0, p = 0;
        uint64_t tgt = ~0ull, ebase = 0, pm = 1ull << 63;
        int pe = 0;
        if (act) {
            d = perm ? order[(int)(nl & (n_ord - 1)) * ND + v] : order[v];
            p = perm ? v : phase_of[v];
            const uint64_t np = (uint64_t)(P.sched_begin + nl) * PART_PHASE_SLOTS + (uint64_t)p;
            ebase = (np << 32) | ((uint64_t)j << 16);
            // target = floor(X M / 2^64), clock variate V 2^-53 as a
            // normalised mantissa pm / 2^63 times 2^pe
            const uint4 w = kmcdev::philox4x32_10(
                make_uint4((uint32_t)j, (uint32_t)d, (uint32_t)np, (uint32_t)(np >> 32) & 0xFFFFFFu), key);
            tgt = __umul64hi(((uint64_t)w.y << 32) | w.x, M);
            const uint64_t V = ((((uint64_t)w.w << 32) | w.z) >> 11) + 1ull;
            const int z = __clzll((long long)V);
            pm = V << z;
            pe = 10 - z;
        }
        // does a pass with a record end at this lane's step?  (a pass ends with
        // the last step of its last visit)
        int64_t rec = -1;
        bool any_rec = false;
        if (want) {
            if (act && j == k - 1 && v - p * dpp == dpp - 1) {
                const int64_t pass = nl * nph + p + 1;
                if (pass % P.obs_every == 0) rec = pass / P.obs_every - 1;
            }
            any_rec = __any_sync(FULL_WARP, rec >= 0);
        }
        if (EXPO) {
            if (any_rec) {
                join(); // everything before this window; then the inclusive products of its steps
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint64_t m2 = __shfl_up_sync(FULL_WARP, pm, off);
                    const int e2 = __shfl_up_sync(FULL_WARP, pe, off);
                    if (lane >= off) kmcdev::mant_mul32(pm, pe, m2, e2);
                }
            } else {
                int e = 0;
                kmcdev::mant_mul32(lM, e, pm, pe);
                lE += e;
            }
        }
        // the real events of the window, in step order
        int pos = 0;
        while (true) {
            // the cumulative class rates of this lane's domain
            uint64_t C[10];
            {
                const uint4 n0 = *reinterpret_cast<const uint4 *>(dcount + d * 12);
                const uint4 n1 = *reinterpret_cast<const uint4 *>(dcount + d * 12 + 4);
                const uint2 n2 = *reinterpret_cast<const uint2 *>(dcount + d * 12 + 8);
                const uint32_t n[10] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w, n2.x, n2.y};
                uint64_t w[10];
#pragma unroll
                for (int c = 0; c < 10; ++c) w[c] = (uint64_t)n[c] * A[c];
                // prefix sums in a shallow tree (pairs, then a chain over pairs)
                const uint64_t s23 = w[2] + w[3], s45 = w[4] + w[5], s67 = w[6] + w[7], s89 = w[8] + w[9];
                C[0] = w[0];
                C[1] = w[0] + w[1];
                C[2] = C[1] + w[2];
                C[3] = C[1] + s23;
                C[4] = C[3] + w[4];
                C[5] = C[3] + s45;
                C[6] = C[5] + w[6];
                C[7] = C[5] + s67;
                C[8] = C[7] + w[8];
                C[9] = C[7] + s89;
            }
            const unsigned real = __ballot_sync(FULL_WARP, lane >= pos && tgt < C[9]);
            if (!real) break;
            const int jx = __ffs(real) - 1;
            // each lane's class (the first c with target < C_c) and member index
            // jj = floor((target - C_{c-1}) / A_c) < n_c: the high word of
            // (target - C_{c-1}) floor((2^64 - 1) / A_c) is jj or jj - 1
            int c = 0;
            uint64_t Cprev = 0;
#pragma unroll
            for (int cc = 0; cc < 9; ++cc) {
                const bool past = tgt >= C[cc];
                c += past ? 1 : 0;
                Cprev = past ? C[cc] : Cprev;
            }
            const ulonglong2 am = atab[c];
            const uint64_t xq = tgt - Cprev;
            uint32_t jj = (uint32_t)__umul64hi(xq, am.y);
            jj = (xq - (uint64_t)jj * am.x >= am.x) ? jj + 1u : jj;
            const uint32_t pick = __shfl_sync(FULL_WARP, (uint32_t)c | ((uint32_t)d << 4) | (jj << 10), jx);
            const uint64_t ev = __shfl_sync(FULL_WARP, ebase, jx);
            const int ec = (int)(pick & 15u), ed = (int)((pick >> 4) & 63u);
            const uint32_t ejj = pick >> 10;
            const int x0 = org[2 * ed], y0 = org[2 * ed + 1];
            // the row of the jj-th member of class c in row-major order: lane l
            // holds the counts of domain rows rpl l .. rpl l + rpl - 1, a byte each
            uint4 rw = make_uint4(0u, 0u, 0u, 0u);
            if (use_rc) {
                if (16 * lane < Hd) rw = *reinterpret_cast<const uint4 *>(rc + (ed * 10 + ec) * Hp + 16 * lane);
            } else {
                const u128 DM = DM0 << x0;
                for (int t = 0; t < 4; ++t) {
                    const int yy = 4 * lane + t;
                    if (yy < Hd)
                        rw.x |= (uint32_t)popc128(class_mask(row_planes(rows, y0 + yy, L, Lm, DM), ec)) << (8 * t);
                }
            }
            const uint32_t q0 = __dp4a(rw.x, 0x01010101u, 0u), q1 = __dp4a(rw.y, 0x01010101u, q0),
                           q2 = __dp4a(rw.z, 0x01010101u, q1), cl = __dp4a(rw.w, 0x01010101u, q2);
            uint32_t incl = cl;
            for (int off = 1; rpl * off < Hd; off <<= 1) {
                const uint32_t u = __shfl_up_sync(FULL_WARP, incl, off);
                if (lane >= off) incl += u;
            }
            uint32_t rr = ejj - (incl - cl);
            const unsigned win = __ballot_sync(FULL_WARP, ejj < incl && rr < cl);
            if (!win) {
                if (lane == 0) atomicOr(P.err, 2);
                pos = jx + 1;
                continue;
            }
            uint32_t yr;
            {
                const bool g0 = rr >= q0, g1 = rr >= q1, g2 = rr >= q2;
                const uint32_t w = g2 ? rw.w : g1 ? rw.z : g0 ? rw.y : rw.x;
                rr -= g2 ? q2 : g1 ? q1 : g0 ? q0 : 0u;
                const uint32_t b0 = w & 255u, b1 = b0 + ((w >> 8) & 255u), b2 = b1 + ((w >> 16) & 255u);
                const bool h0 = rr >= b0, h1 = rr >= b1, h2 = rr >= b2;
                rr -= h2 ? b2 : h1 ? b1 : h0 ? b0 : 0u;
                const int t = 4 * ((g0 ? 1 : 0) + (g1 ? 1 : 0) + (g2 ? 1 : 0)) + (h0 ? 1 : 0) + (h1 ? 1 : 0) + (h2 ? 1 : 0);
                yr = __shfl_sync(FULL_WARP, (uint32_t)(rpl * lane + t) | (rr << 8), __ffs(win) - 1);
            }
            const int yy = (int)(yr & 255u), y = y0 + yy;
            rr = yr >> 8;
            const int ym = (y == 0) ? L - 1 : y - 1, yp = (y == L - 1) ? 0 : y + 1;
            // its column: the row's class mask, 32 columns at a time, the same in
            // every lane; lane i tests whether its column is member rr
            int x = x0;
            for (int t0 = 0; t0 < W; t0 += 32) {
                const int X = x0 + t0, i = X >> 5, sft = X & 31; // bit X: column X - 1
                auto window = [&](int yq, uint32_t &lo, uint32_t &hi) {
                    const uint32_t *w = rows + PART_ROW32 * yq + i;
                    const uint32_t a0 = w[0], a1 = w[1], a2 = w[2]; // i <= 3
                    lo = __funnelshift_r(a0, a1, sft);
                    hi = __funnelshift_r(a1, a2, sft);
                };
                uint32_t cl0, cl1, nl0, nl1, sl0, sl1;
                window(y, cl0, cl1);
                window(ym, nl0, nl1);
                window(yp, sl0, sl1);
                const uint32_t wn = cl0, cc = __funnelshift_r(cl0, cl1, 1), en = __funnelshift_r(cl0, cl1, 2);
                const uint32_t nn = __funnelshift_r(nl0, nl1, 1), ss = __funnelshift_r(sl0, sl1, 1);
                const uint32_t s1 = nn ^ ss, c1 = nn & ss, s2 = wn ^ en, c2 = wn & en, u0 = s1 & s2;
                const uint32_t b0 = s1 ^ s2, b1 = c1 ^ c2 ^ u0, b2 = (c1 & c2) | (c1 & u0) | (c2 & u0);
                const int q = (ec >= 5) ? ec - 5 : ec;
                const uint32_t diff = (b2 ^ ((q & 4) ? ~0u : 0u)) | (b1 ^ ((q & 2) ? ~0u : 0u)) | (b0 ^ ((q & 1) ? ~0u : 0u));
                const uint32_t cols = (W - t0 >= 32) ? ~0u : ((1u << (W - t0)) - 1u);
                const uint32_t mk = (ec >= 5 ? cc : ~cc) & ~diff & cols;
                const uint32_t pc = (uint32_t)__popc(mk);
                const unsigned it = __ballot_sync(FULL_WARP, ((mk >> lane) & 1u) && (uint32_t)__popc(mk & ((1u << lane) - 1u)) == rr);
                x = X + max(__ffs(it) - 1, 0);
                if (rr < pc) break;
                rr -= pc;
            }
            // the flip changes the classes of the site and its four
            // neighbours (lanes 0..4: site, W, E, N, S): the site's spin, and
            // every neighbour's count by one (by two on a 2 x 2 lattice, whose
            // opposite neighbours are the same site)
            int sx = x + dxl, sy = y + dyl, syy = yy + dyl;
            const int bx = x - x0 + dxl;
            const bool cross = bx < 0 || bx == W || syy < 0 || syy == Hd;
            const int sd = cross ? nbd[4 * ed + ((lane + 3) & 3)] : ed;
            sx = (sx < 0) ? L - 1 : (sx == L) ? 0 : sx;
            sy = (sy < 0) ? L - 1 : (sy == L) ? 0 : sy;
            syy = (syy < 0) ? Hd - 1 : (syy == Hd) ? 0 : syy;
            const bool mine = lane < 5 && !(L == 2 && (lane == 2 || lane == 4));
            const int gain = (ec < 5) ? 1 : -1;
            const int old_c = site_class(rows, sx, sy, (sy == 0) ? L - 1 : sy - 1, (sy == L - 1) ? 0 : sy + 1);
            const int new_c = (lane == 0) ? old_c + 5 * gain : old_c + (L == 2 ? 2 : 1) * gain;
            __syncwarp();
            if (mine) {
                atomicSub(&dcount[sd * 12 + old_c], 1u);
                atomicAdd(&dcount[sd * 12 + new_c], 1u);
                if (use_rc) {
                    const int i0 = (sd * 10 + old_c) * Hp + syy, i1 = (sd * 10 + new_c) * Hp + syy;
                    atomicSub(reinterpret_cast<unsigned *>(rc) + (i0 >> 2), 1u << (8 * (i0 & 3))); // the byte holds this site
                    atomicAdd(reinterpret_cast<unsigned *>(rc) + (i1 >> 2), 1u << (8 * (i1 & 3)));
                }
            }
            if (lane == 0) {
                // the site's bit and its copy at the other end of the row
                uint32_t *w = rows + PART_ROW32 * y;
                w[(x + 1) >> 5] ^= 1u << ((x + 1) & 31);
                if (x == 0) w[(L + 1) >> 5] ^= 1u << ((L + 1) & 31);
                if (x == L - 1) w[0] ^= 1u;
            }
            __syncwarp();
            H = (H ^ (ev | (uint64_t)(yy * W + (x - x0)))) * HASH_PRIME;
            ++flips;
            // flipping spin s with neighbour sum 2 q - 4 changes the bond sum by
            // -2 s (2 q - 4) and the magnetisation by -2 s, for every record from
            // this step on
            if (lane >= jx) {
                bonds += 2 * gain * (2 * (ec < 5 ? ec : ec - 5) - 4);
                mag += 2 * gain;
            }
            pos = jx + 1;
        }
        if (want) {
            if (rec >= 0) {
                uint64_t cm = clkM;
                int64_t ce = clkE;
                if (EXPO) kmcdev::mant_mul(cm, ce, pm, (int64_t)pe);
                write_record(rec, bonds, mag, cm, ce, steps0 + s0 + lane + 1);
            }
            bonds = __shfl_sync(FULL_WARP, bonds, 31);
            mag = __shfl_sync(FULL_WARP, mag, 31);
            if (EXPO && any_rec)
                kmcdev::mant_mul(clkM, clkE, __shfl_sync(FULL_WARP, pm, 31), (int64_t)__shfl_sync(FULL_WARP, pe, 31));
        }
        j += jump_j;
        const int carry = (j >= k) ? 1 : 0;
        j -= carry ? k : 0;
        v += jump_v + carry;
        nl += jump_n;
        if (v >= Vs) {
            v -= Vs;
            ++nl;
        }
    }
    if (EXPO) join();
    if (k == 0 && want) {
        // visits without steps: every record holds the state as it is
        for (int64_t rec = lane; rec < P.n_sched * nph / P.obs_every; rec += 32)
            write_record(rec, bonds, mag, clkM, clkE, steps0);
    }

    // write the lattice back
    __syncwarp();
    int8_t *out = P.spins + (size_t)tr * L * L;
    for (int y = 0; y < L; ++y) {
        for (int x = lane; x < L; x += 32)
            out[(size_t)y * L + x] = ((rows[PART_ROW32 * y + ((x + 1) >> 5)] >> ((x + 1) & 31)) & 1u) ? (int8_t)1 : (int8_t)-1;
    }
    if (lane == 0) {
        P.hash[tr] = H;
        P.clkM[tr] = clkM;
        P.clkE[tr] = clkE;
        P.flips[tr] = flips;
        P.steps[tr] = steps0 + total;
        P.t[tr] = kmcdev::domain_time(EXPO, clkM, clkE, steps0 + total, __dmul_rn(N, P.nu));
    }
}

} // namespace kmcpart
