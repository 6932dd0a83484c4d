// kmc_ring.cuh -- sm_103a device code of the 1D ring (Sec. 3.1): many
// independent trajectories of an N_S-spin toroidal Ising ring (N_S <= 64),
// cut into N_D contiguous domains of L_d spins (Sec. 3.1, Eq. 1D partitions),
// each domain process k uniformised steps with its two halo spins frozen.
//
// Data parallelism is over trajectories (the paper's N_TRAJ independent
// runs per setting, Eq. time dependent averages): one thread owns one
// trajectory for the whole launch, its configuration one register word
// (bit n set iff spin n is up).  Within a thread the domain processes of a
// schedule run in schedule order, so the halo of a visit is the live word:
// no other domain of the trajectory moves while it runs.  Observation records
// per trajectory are coalesced stores; the ensemble sums over trajectories
// (integers, so their order does not matter) are reduced per warp with
// ballots and warp reductions and added to global memory with one atomic per
// warp and quantity.
//
// What bounds it: integer issue and the fixed latency between dependent
// instructions.  48000 trajectories of 8 spins are 2.4 warps per scheduler;
// ncu counts 49 % of the issue slots used, the ALU pipe 46 % and the multiply
// pipe 40 % busy, stalls led by fixed-latency waits.  A warp runs the event
// path whenever one of its 32 trajectories has an event, so a step is kept
// short rather than skipped: the visit works on a 32-bit window of its domain
// (below), and the next step's Philox block, which depends on nothing, is
// drawn in line with the event so that its multiplies fill the event's waits.
// Measured against a step of draw, then event, on 64-bit words: 48000 x 8
// spins, k = 5, 40 sweeps with ensemble sums 1031 -> 732 us; 6000 x 64 spins,
// k = 10, 10 sweeps with records 931 -> 651 us.
#pragma once

#include <cstdint>

#include "kmc_kernels.cuh"

namespace kmcring {

using kmcdev::FULL_WARP;
using kmcdev::HASH_PRIME;

constexpr int RING_CLASSES = 6;      // c = 3*up + (number of up neighbours)
constexpr int RING_PHASE_SLOTS = 64; // Philox phase index np = n*64 + p
constexpr int RING_ENS_FIXED = 4;    // sum bonds, sum mag, sum bonds*mag, sum mag^2; then per-site up counts
constexpr int RING_BLOCK = 64;
constexpr uint32_t RING_TAG_PERM = 2u;

struct RingParams {
    int n_traj, NS, Ld, k;
    int schedule;         // KMC_SCHED_*
    int obs_every;        // passes between records (0: none)
    int64_t sched_begin, n_sched;
    double J, nu;
    const uint64_t *seed; // [n_traj]
    const uint64_t *A;    // [n_traj][6] fixed-point acceptance, P = 63 - log2(L_d)
    const double *h;      // [n_traj]
    uint64_t *state, *hash, *clkM;
    int64_t *clkE, *flips, *steps;
    double *t;            // [n_traj] clock after the launch
    double *obs;          // [n_rec][n_traj][4] or null
    uint64_t *obs_state;  // [n_rec][n_traj] or null
    unsigned long long *ens; // [n_rec][4 + NS] or null (added to)
};

// A visit works on its domain alone: its spins and its two halo spins as a
// window of 32 bits (domains of up to 32 spins; half the instructions of
// every mask, shift and bit count), else of 64.
__device__ __forceinline__ int ring_popc(uint32_t v) { return __popc(v); }
__device__ __forceinline__ int ring_popc(uint64_t v) { return __popcll(v); }

// Position of the rr-th (0-based) set bit of m, a window of Ld bits; rr < popc(m).
__device__ __forceinline__ int ring_select(uint64_t m, uint32_t rr, int) { return kmcdev::select_bit(m, rr); }
__device__ __forceinline__ int ring_select(uint32_t w, uint32_t rr, int Ld)
{
    int pos = 0;
    uint32_t c;
    if (Ld > 8) { // (the same in every lane)
        c = __popc(w & 0xFFFFu);
        if (rr >= c) { rr -= c; w >>= 16; pos += 16; }
        c = __popc(w & 0xFFu);
        if (rr >= c) { rr -= c; w >>= 8; pos += 8; }
    }
    c = __popc(w & 0xFu);  if (rr >= c) { rr -= c; w >>= 4; pos += 4; }
    c = __popc(w & 0x3u);  if (rr >= c) { rr -= c; w >>= 2; pos += 2; }
    if (rr >= (w & 1u)) pos += 1;
    return pos;
}

// The left neighbours of a ring of NS bits: bit n is spin n-1.
__device__ __forceinline__ uint64_t ring_left(uint64_t S, int NS, uint64_t NM)
{
    return ((S << 1) | (S >> (NS - 1))) & NM;
}

// Inclusive cumulative rates C_c = sum_{c' <= c} n_c' A_c' in class order 0..5
// of a domain of Ld spins (s; DM: its sites), with the spins left of bit 0
// and right of bit Ld - 1 (hl, hr), and the words that hold the neighbours.
template <typename word>
__device__ __forceinline__ void ring_cumulative(uint64_t (&C)[RING_CLASSES], word &lw, word &rw, word s, word hl, word hr,
                                                int Ld, word DM, const uint64_t (&A)[RING_CLASSES])
{
    lw = (word)(s << 1) | hl;
    rw = (s >> 1) | (word)(hr << (Ld - 1));
    const word q0 = ~(lw | rw), q1 = lw ^ rw, q2 = lw & rw;
    const word dn = ~s & DM;
    const word M[RING_CLASSES] = {dn & q0, dn & q1, dn & q2, s & q0, s & q1, s & q2};
    uint64_t acc = 0;
#pragma unroll
    for (int c = 0; c < RING_CLASSES; ++c) {
        acc += (uint64_t)(uint32_t)ring_popc(M[c]) * A[c];
        C[c] = acc;
    }
}

// One step's random numbers: its target, and its clock variate V 2^-53.
struct RingDraw {
    uint64_t tgt, V;
};
__device__ __forceinline__ RingDraw ring_draw(uint32_t j, uint32_t d, uint64_t np, uint2 key)
{
    const uint4 w = kmcdev::philox4x32_10(make_uint4(j, d, (uint32_t)np, (uint32_t)(np >> 32) & 0xFFFFFFu), key);
    return {(((uint64_t)w.y << 32) | w.x) >> 1, ((((uint64_t)w.w << 32) | w.z) >> 11) + 1ull};
}

// One domain process: domain d, k steps of global phase np.  Step j draws
// Philox {j, d, np_lo, np_hi} with the trajectory seed: target = (w0 |
// w1<<32) >> 1 on [0, L_d 2^P); target >= R' is a null step; otherwise the
// class is the first c with target < C_c and the member jj = (target -
// C_{c-1}) / A_c, counted in ascending site order, flips (App. A, the
// n-fold way's cumulative selection of Sec. 2.1).  jj < n_c <= 64: an FP32
// estimate with every rounding toward the lower side (x down, A_c up, the
// reciprocal down, the product toward zero) is jj or jj - 1, and one exact
// integer comparison decides.  The 32 trajectories of a warp step together;
// the next step's draw does not depend on this step's event, so the two stand
// in one straight line and fill each other's latencies, and a trajectory
// without an event runs it without effect.  `cur` is the draw of step 0 on
// entry and, with `more`, that of the next visit's (domain d2, phase np2) on
// return; a variate enters the clock with its step.
template <bool EXPO, typename word>
__device__ __forceinline__ void ring_visit(uint64_t &S, uint64_t &H, int64_t &flips, uint64_t &clkM, int64_t &clkE, int d,
                                           int Ld, int k, int NS, word DM, uint64_t np, uint2 key,
                                           const uint64_t (&A)[RING_CLASSES], const float (&invA)[RING_CLASSES],
                                           unsigned lanes, RingDraw &cur, bool more, int d2, uint64_t np2)
{
    const int first = d * Ld;
    const word s0 = (word)(S >> first) & DM;
    word s = s0;
    // the halo spins; the only domain of a ring is its own neighbour
    const bool own = Ld == NS;
    word hl = (word)(S >> (first == 0 ? NS - 1 : first - 1)) & 1, hr = (word)(S >> (first + Ld == NS ? 0 : first + Ld)) & 1;
    uint64_t C[RING_CLASSES];
    word lw, rw;
    ring_cumulative(C, lw, rw, s, hl, hr, Ld, DM, A);
    auto step = [&](int j, auto draw_next) {
        const uint64_t tgt = cur.tgt;
        const bool ev = tgt < C[RING_CLASSES - 1]; // else a null step
        if (EXPO) {
            const int z = __clzll((long long)cur.V);
            kmcdev::mant_mul(clkM, clkE, cur.V << z, (int64_t)(10 - z));
        }
        draw_next();
        if (__any_sync(lanes, ev)) {
            uint64_t lo = 0, Ac = A[0];
            float inv = invA[0];
            int c = 0;
#pragma unroll
            for (int cc = 1; cc < RING_CLASSES; ++cc) {
                const bool past = tgt >= C[cc - 1];
                lo = past ? C[cc - 1] : lo;
                Ac = past ? A[cc] : Ac;
                inv = past ? invA[cc] : inv;
                c = past ? cc : c;
            }
            const uint64_t x = tgt - lo;
            uint32_t jj = (uint32_t)__fmul_rz(kmcdev::u64_to_float_rz(x), inv);
            jj = (x - (uint64_t)jj * Ac >= Ac) ? jj + 1u : jj;
            const int q = (c >= 3) ? c - 3 : c;
            const word qm = (q == 0) ? ~(lw | rw) : ((q == 1) ? (lw ^ rw) : (lw & rw));
            const int site = ring_select((word)(((c >= 3) ? s : ~s) & qm & DM), jj, Ld) & (int)(8 * sizeof(word) - 1);
            s ^= ev ? (word)1 << site : (word)0;
            if (own) {
                hl = s >> (Ld - 1);
                hr = s & 1;
            }
            flips += ev ? 1 : 0;
            const uint64_t h = (H ^ ((np << 32) | ((uint64_t)j << 16) | (uint64_t)site)) * HASH_PRIME;
            H = ev ? h : H;
            ring_cumulative(C, lw, rw, s, hl, hr, Ld, DM, A);
        }
    };
    // (the last step stands by itself: the draws of the others are all of this
    // visit's domain and phase, whose share of the first Philox round then is
    // formed once; with one loop that chose per step 770 and 737 us)
    for (int j = 0; j + 1 < k; ++j) step(j, [&]() { cur = ring_draw((uint32_t)(j + 1), (uint32_t)d, np, key); });
    step(k - 1, [&]() { if (more) cur = ring_draw(0u, (uint32_t)d2, np2, key); });
    S ^= (uint64_t)(s ^ s0) << first;
}

// Uniform random order of the n_dom domains of schedule n (the paper's
// random schedule per sweep): Fisher-Yates, draw i (n_dom-1 down to 1) from
// Philox {i, 0, n_lo, n_hi | TAG_PERM << 24}: position i swaps with
// floor(x (i+1) / 2^64), x = w0 | w1 << 32.  Up to 16 domains: the order is 16
// nibbles in a register; more: bytes in local memory.
struct RingOrder {
    uint64_t nib;
    uint8_t order[64];
    __device__ __forceinline__ void shuffle(int n_dom, uint64_t n, uint2 key)
    {
        nib = 0xFEDCBA9876543210ull;
        if (n_dom > 16)
            for (int i = 0; i < n_dom; ++i) order[i] = (uint8_t)i;
        for (int i = n_dom - 1; i >= 1; --i) {
            const uint4 w = kmcdev::philox4x32_10(
                make_uint4((uint32_t)i, 0u, (uint32_t)n, ((uint32_t)(n >> 32) & 0xFFFFFFu) | (RING_TAG_PERM << 24)), key);
            const uint64_t x = ((uint64_t)w.y << 32) | w.x;
            const int jx = (int)__umul64hi(x, (uint64_t)(i + 1));
            if (n_dom > 16) {
                const uint8_t t = order[i];
                order[i] = order[jx];
                order[jx] = t;
            } else {
                const uint64_t dif = ((nib >> (4 * i)) ^ (nib >> (4 * jx))) & 0xFull;
                nib ^= (dif << (4 * i)) ^ (dif << (4 * jx));
            }
        }
    }
    __device__ __forceinline__ int at(int n_dom, int p) const
    {
        return n_dom > 16 ? order[p] : (int)((nib >> (4 * p)) & 0xFull);
    }
};

// Clock of a trajectory: the mean over domains of t_d (Sec. 2.1), i.e.
// -ln(product of all its variates) / (N_S nu) (exponential) or
// steps / (N_S nu) (expected).
__device__ __forceinline__ double ring_clock(bool expo, uint64_t M, int64_t E, int64_t steps, int NS, double nu)
{
    return kmcdev::domain_time(expo, M, E, steps, __dmul_rn((double)NS, nu));
}

// Two warps per CTA: a CTA's trajectories need nothing of each other (the
// ensemble sums go out by warp), and small CTAs load the SMs evenly (48000
// trajectories are 9.9 warps per SM; CTAs of 4 warps put 12 on some and 8 on
// others).
template <bool EXPO, typename word>
__global__ void __launch_bounds__(RING_BLOCK, 8) ring_kernel(const RingParams P)
{
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const bool active = tid < P.n_traj;
    const int r = active ? tid : 0;
    const int NS = P.NS, Ld = P.Ld, ND = NS / Ld, k = P.k;
    const int n_ens = RING_ENS_FIXED + NS;
    constexpr int WB = 8 * (int)sizeof(word);
    const uint64_t NM = (NS == 64) ? ~0ull : ((1ull << NS) - 1ull);
    const word DM = (Ld == WB) ? ~(word)0 : (((word)1 << (Ld & (WB - 1))) - (word)1);

    uint64_t A[RING_CLASSES];
    float invA[RING_CLASSES]; // 1/A_c from below: A_c rounded up, reciprocal rounded down
#pragma unroll
    for (int c = 0; c < RING_CLASSES; ++c) {
        A[c] = P.A[(size_t)r * RING_CLASSES + c];
        invA[c] = A[c] ? __frcp_rd(kmcdev::u64_to_float_ru(A[c])) : 0.0f;
    }
    const uint64_t seed = P.seed[r];
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    const double hr = P.h[r];
    uint64_t S = P.state[r], H = P.hash[r], clkM = P.clkM[r];
    int64_t clkE = P.clkE[r], flips = P.flips[r], steps = P.steps[r];

    const bool perm = P.schedule == kmcdev::SCHED_RANDOM_PERM;
    const int ncol = (ND == 1) ? 1 : 2;
    const int nph = perm ? ND : (P.schedule == kmcdev::SCHED_PALINDROME ? 2 * ncol : ncol);
    const unsigned lanes = __ballot_sync(FULL_WARP, active);
    RingOrder order;
    RingDraw cur = {0, 0};
    int64_t rec = 0;
    int until = P.obs_every; // passes before the next record
    for (int64_t nl = 0; nl < P.n_sched; ++nl) {
        const uint64_t n = (uint64_t)(P.sched_begin + nl);
        if (perm && active) order.shuffle(ND, n, key);
        for (int p = 0; p < nph; ++p) {
            const uint64_t np = n * RING_PHASE_SLOTS + (uint64_t)p;
            if (active && k > 0) {
                if (perm) {
                    // the next visit is known up to the end of the sweep
                    const int d = order.at(ND, p);
                    if (p == 0) cur = ring_draw(0u, (uint32_t)d, np, key);
                    const bool more = p + 1 < nph;
                    ring_visit<EXPO>(S, H, flips, clkM, clkE, d, Ld, k, NS, DM, np, key, A, invA, lanes, cur, more,
                                     more ? order.at(ND, p + 1) : 0, np + 1);
                    steps += k;
                } else {
                    // colour of phase p: 0 1 [1 0] (one colour when N_D = 1)
                    auto colour = [&](int q) { return (q < ncol) ? q : (2 * ncol - 1 - q); };
                    if (p == 0 && nl == 0) cur = ring_draw(0u, 0u, np, key);
                    for (int d = colour(p); d < ND; d += ncol) {
                        const bool stay = d + ncol < ND, turn = p + 1 == nph;
                        const bool more = stay || !turn || nl + 1 < P.n_sched;
                        ring_visit<EXPO>(S, H, flips, clkM, clkE, d, Ld, k, NS, DM, np, key, A, invA, lanes, cur, more,
                                         stay ? d + ncol : turn ? 0 : colour(p + 1),
                                         stay ? np : turn ? (n + 1) * RING_PHASE_SLOTS : np + 1);
                        steps += k;
                    }
                }
            }
            if (P.obs_every > 0 && --until == 0) {
                until = P.obs_every;
                // bonds = sum_n s_n s_{n+1}: NS - 2 * (number of unlike neighbour pairs)
                const int unlike = __popcll((S ^ ring_left(S, NS, NM)) & NM);
                const int bonds = NS - 2 * unlike;
                const int mag = 2 * __popcll(S & NM) - NS;
                if (active) {
                    const size_t o = (size_t)rec * P.n_traj + r;
                    if (P.obs) {
                        const double e = __ddiv_rn(__dsub_rn(__dmul_rn(-P.J, (double)bonds), __dmul_rn(hr, (double)mag)),
                                                   (double)NS);
                        const double m = __ddiv_rn((double)mag, (double)NS);
                        double4_32a v;
                        v.x = e;
                        v.y = m;
                        v.z = __dmul_rn(e, m);
                        v.w = ring_clock(EXPO, clkM, clkE, steps, NS, P.nu);
                        reinterpret_cast<double4_32a *>(P.obs)[o] = v;
                    }
                    if (P.obs_state) P.obs_state[o] = S;
                }
                if (P.ens != nullptr) {
                    // ensemble sums over the warp, lane i adding quantity i, i + 32, ...
                    __syncwarp();
                    const int b = active ? bonds : 0, m = active ? mag : 0;
                    const int s0 = __reduce_add_sync(FULL_WARP, b);
                    const int s1 = __reduce_add_sync(FULL_WARP, m);
                    const int s2 = __reduce_add_sync(FULL_WARP, b * m);
                    const int s3 = __reduce_add_sync(FULL_WARP, m * m);
                    unsigned long long *ens = P.ens + (size_t)rec * n_ens;
                    int mine = (lane == 0) ? s0 : (lane == 1) ? s1 : (lane == 2) ? s2 : s3;
                    for (int q = 0; q < n_ens; q += 32) {
                        for (int i = (q == 0 ? RING_ENS_FIXED : 0); i < 32 && q + i < n_ens; ++i) {
                            const int site = q + i - RING_ENS_FIXED;
                            const int cnt = __popc(__ballot_sync(FULL_WARP, active && ((S >> site) & 1ull)));
                            if (lane == i) mine = cnt;
                        }
                        if (q + lane < n_ens && mine != 0) atomicAdd(&ens[q + lane], (unsigned long long)(long long)mine);
                    }
                }
                ++rec;
            }
        }
    }
    if (active) {
        P.state[r] = S;
        P.hash[r] = H;
        P.clkM[r] = clkM;
        P.clkE[r] = clkE;
        P.flips[r] = flips;
        P.steps[r] = steps;
        P.t[r] = ring_clock(EXPO, clkM, clkE, steps, NS, P.nu);
    }
}

} // namespace kmcring
