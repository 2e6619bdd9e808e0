// Joint recurrence over the device-group state as a search for the bottleneck (sm_100a).
//
// The smallest bottleneck over all stage-type sequences of a configuration is the smallest B for which some sequence has a
// partition without a stage above B.  For a given B a state u (stages of each type placed) with last type t needs one bit
// per end layer instead of a value:
//     reach[u][t] = OR over stage lengths n, OR over types t' of the stage before,
//                   (reach[u - e_t][t'] AND ok[t][t'][n]) << n
// where bit k of ok says that layers (k, k + n] on type t cost at most B behind a stage of type t' and fit the memory of
// this depth.  All bits of a state sit in one to three 64-bit words (bits count from the smallest end layer of the level), so
// a level of every state takes a few logic instructions per (type, type before, length) and both levels of the recurrence
// stay in shared memory.  The stage costs are finitely many numbers: after a test, B moves to the nearest of them, so the
// bisection ends after about a dozen tests, each exact.  It starts at a guess: the B at which stages of mean cost would add up
// to all layers (capacity); the answer lies within 2 % of it for half of the configurations, within 30 % for nine in ten.
//
// Lengths whose masks are full at a depth (most, once B is near the answer) need no mask at all.
//
// 1,024 devices, 3,114 homogeneous configurations of up to 3,825 states: 38.4 ms with a value per end layer in global memory,
// 2.83 ms in this form, 2.17 ms since the tests start at the guess instead of a lower bound (12 tests a feasible configuration
// instead of 16 to 18), lengths are summed up in one direction and transfers that cannot occur are left out.  Five blocks an SM
// instead of four (48 registers a thread, spilled): 2.36 ms.  128 threads a block: 3.6 ms, 192: 3.2 ms against 2.83 (few
// configurations are feasible, and each is a chain of levels and tests); a lane for all next types of a state instead of one: 4.4 ms.
// Measured on other tables, where this form took 2.40 ms: a warp that keeps to one type 2.50 (types of long stages hold up the
// others); first a search with the least transfer of each type, whose states need no type before, 2.72 (its tests cost as much).
//
// One block per configuration.  Bound by instruction issue of the level loop: per (state, type) four logic operations per
// (type before, length), and by the barrier of each level.  The value form -- a 64-bit minimum per end layer and split, rows in
// global memory -- is kept for classes whose bits or masks do not fit (joint_dp_kernel).
#pragma once
#include "hap_device.cuh"

namespace hap {

constexpr int kReachThreads = 256;
constexpr int kReachWords = 3;                    // 64-bit words of a state at most
constexpr int kReachKc = 2 + HAP_MAX_TYPES;       // transfer into a stage: same type intra / inter node, from type 0..3
constexpr int kReachOk = 2 * HAP_MAX_TYPES;       // masks of a (depth, type, length): [same-type link][type before]

struct JointReach {
    int PP, lmax, words;                          // stages; most states of a level; 64-bit words per state and type
    int nwin;                                     // most stage lengths of a type
    int nmin[HAP_MAX_TYPES], nmax[HAP_MAX_TYPES], cnt[HAP_MAX_TYPES];
    int fin[HAP_MAX_TYPES];                       // slot, at level PP - 1, of "one stage of type t left"
    unsigned id_lo, n_ids;                        // its configurations in the id list
    unsigned first[HAP_MAX_TYPES];                // slot, at level 1, of "one stage of type t placed"
    unsigned ent_off[HAP_MAX_PP + 1];             // level i's entries: [type][state] slot before | type << 16 | same-type link << 18 | valid << 19
    unsigned n_states[HAP_MAX_PP + 1];
    int base[HAP_MAX_PP + 1], width[HAP_MAX_PP + 1];      // end layer of bit 0; bits
    const unsigned *ent;
};

// Which limits are tested, and when the answer is known.  The answer lies between lo (no smaller stage cost can do) and hi (does; kInf:
// not known that any does).  From a guess on in steps that double while they are taken, then halfway; whether anything is feasible at all
// is asked once three tests have failed, or first where that is in doubt.  An answer under a larger choice of levels is tested before that:
// mostly it remains.
// Every limit lies in [lo, hi): a step is taken only where it is shorter than the way to the halving point, and never again once it was
// not, so that it neither overflows nor leaves the interval, and each test makes that smaller -- whatever the stage costs are, those
// beyond the supported range included.  At most 128 tests: 62 steps, 62 halvings, the larger choice's answer, the largest limit, one of each that
// is not taken.
struct LimitSearch {
    enum Way { kHalve, kUp, kDown };
    i64 lo, hi, B, step, guess;                   // B: the limit to be tested
    int way, failed;
    bool at_floor, doubt;                         // B is the answer under a larger choice of levels; nothing may be feasible, not asked yet

    // low: a lower bound on the answer; floor_b: the answer under a larger choice of levels (0: none); mean: the guess; doubtful: whether
    // anything is feasible is to be asked first
    __host__ __device__ void begin(i64 low, i64 floor_b, i64 mean, bool doubtful)
    {
        lo = low > floor_b ? low : floor_b; hi = kInf;
        at_floor = floor_b > 0 && lo == floor_b;
        guess = mean > lo && mean < kInf ? mean : lo;
        way = kUp; failed = 0; step = guess / 64 + 1;
        doubt = doubtful && lo < kInf - 1;
        B = at_floor ? lo : doubt ? kInf - 1 : guess;
    }

    // Whether B can do, and the nearest stage costs: the largest at most B, the smallest above (kInf: none).  False: the answer is lo (kInf: infeasible).
    __host__ __device__ bool next(bool can, i64 dn, i64 up)
    {
        if (can && at_floor) return false;
        if (can) {
            hi = dn < B ? dn : B;
            if (B != kInf - 1) way = way != kHalve && (way == kDown || failed == 0) ? kDown : kHalve;
        } else {
            lo = up > B ? up : B + 1;
            if (lo > kInf) lo = kInf;
            if (!at_floor) { ++failed; if (way == kDown) way = kHalve; }
        }
        if (lo >= hi) return false;               // (a test that succeeds at lo is the answer)
        if (at_floor && doubt) { at_floor = false; B = kInf - 1; return true; }
        if (at_floor || doubt) {                  // the guess, once what came before it is answered
            at_floor = doubt = false;
            B = guess > lo && guess < hi ? guess : lo;
            return true;
        }
        if (hi == kInf && failed == 3) { B = kInf - 1; return true; }
        B = lo + (hi - lo) / 2;
        if (way != kHalve) {
            const i64 room = way == kUp ? B - lo : hi - B;
            if (step < room) { B = way == kUp ? lo + step : hi - step; step *= 2; }
            else way = kHalve;
        }
        return true;
    }
};

template <int W> struct Bits { u64 w[W]; };

template <int W>
__device__ __forceinline__ Bits<W> bits_shift(const Bits<W> &x, int s)      // by s towards higher end layers (s < 0: lower)
{
    Bits<W> y;
    if (W == 1) { y.w[0] = s >= 0 ? (s < 64 ? x.w[0] << s : 0) : (s > -64 ? x.w[0] >> -s : 0); return y; }
    const int r = s >= 0 ? s : -s, words = r >> 6, b = r & 63;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        u64 near = 0, far = 0;                                  // the words that a word takes its bits from
#pragma unroll
        for (int v = 0; v < W; ++v) {
            if (v == (s >= 0 ? w - words : w + words)) near = x.w[v];
            if (v == (s >= 0 ? w - words - 1 : w + words + 1)) far = x.w[v];
        }
        y.w[w] = s >= 0 ? (b ? near << b | far >> (64 - b) : near) : (b ? near >> b | far << (64 - b) : near);
    }
    return y;
}

__host__ __device__ inline int reach_mask_words(int N) { return (N + 31) / 32; }

struct ReachSmem { u32 rows, wa, sk, m, a, reach, span, least, mean, lvl, fin, total; };
__host__ __device__ inline ReachSmem reach_smem(int N, int T, int R, int RW, int PP, int lmax, int nwin, int words)
{
    auto up = [](size_t v) { return (u32)((v + 15) / 16 * 16); };
    const size_t n1 = (size_t)N + 1;
    ReachSmem s;
    size_t o = 0;
    s.rows = (u32)o; o = up(o + (size_t)T * RW * n1 * 8);
    s.wa = (u32)o; o = up(o + 2 * n1 * 8);
    s.sk = (u32)o; o = up(o + n1);
    s.a = (u32)o; o = up(o + (size_t)2 * T * nwin * kReachOk * words * 8);
    s.reach = (u32)o; o = up(o + (size_t)2 * HAP_MAX_TYPES * lmax * words * 8);
    s.m = (u32)o; o = up(o + (size_t)T * nwin * R * kReachKc * reach_mask_words(N) * 4);
    s.span = (u32)o; o = up(o + (size_t)T * nwin * R * 16);
    s.least = (u32)o; o = up(o + (size_t)T * nwin * R * 8);
    s.mean = (u32)o; o = up(o + (size_t)T * nwin * R * 8);
    s.fin = (u32)o; o = up(o + (size_t)T * nwin * 4);
    s.lvl = (u32)o; o = up(o + (size_t)PP * T * nwin);
    s.total = (u32)(o > 0xffffffffull ? 0xffffffffull : o);
    return s;
}

template <bool LINEAR, int W>
__global__ void __launch_bounds__(kReachThreads, W > 2 ? 2 : 4)      // (three words: 85 KB and more of shared memory a block; 1,966 us against 2,368 with four and spilled registers)
joint_reach_kernel(const DevConst dc, const JointReach *classes, int n_classes, const unsigned *ids, const i64 *c2, const i64 *coef, i64 *out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ JointReach jc;
    __shared__ MaskInfo<i64> minfo[kMaxMasks];
    __shared__ i64 sP2P[HAP_MAX_TYPES][6];
    __shared__ i64 szero[1];
    __shared__ u64 s_dn, s_up;                              // bounds that a test leaves: next stage costs around B
    __shared__ int s_enough[kReachThreads / 32], s_spare;
    __shared__ Bits<W> s_level[HAP_MAX_PP + 1];             // all end layers of a level
    __shared__ i64 s_res[HAP_MAX_RC_MASKS];
    __shared__ int s_end[3][HAP_MAX_TYPES], s_full[3][HAP_MAX_TYPES];      // by depth % 3 and type: lengths from s_end on have empty
                                                            // masks, those before s_full have full ones
    __shared__ i64 s_k2[HAP_MAX_TYPES][2], s_kmin[HAP_MAX_TYPES];
    __shared__ u32 s_via[HAP_MAX_TYPES];                    // transfers that can occur into a stage of the type, a bit each
    __shared__ u32 s_used[HAP_MAX_TYPES];                   // per type: levels of stages between the first and the last
    const int tid = threadIdx.x, wib = tid >> 5, lane = tid & 31;
    constexpr int nwarps = kReachThreads / 32;
    const int N = dc.N, T = dc.T, R = dc.R, n1 = N + 1, RW = LINEAR ? R : 2;
    {
        int ci = 0;
        while (ci + 1 < n_classes && blockIdx.x >= classes[ci + 1].id_lo) ++ci;
        static_assert(sizeof(JointReach) % 4 == 0, "copied in words");
        for (int q = tid; q < (int)(sizeof(JointReach) / 4); q += kReachThreads)
            reinterpret_cast<u32 *>(&jc)[q] = reinterpret_cast<const u32 *>(classes + ci)[q];
    }
    const unsigned p = ids[blockIdx.x];
    const hap_pconf pc = dc.pconf[p];
    const int PP = pc.PP;
    __syncthreads();
    const int nwin = jc.nwin, lmax = jc.lmax, mw = reach_mask_words(N);
    const ReachSmem lay = reach_smem(N, T, R, RW, PP, lmax, nwin, W);
    i64 *sR = reinterpret_cast<i64 *>(smem_raw + lay.rows);
    i64 *sW = reinterpret_cast<i64 *>(smem_raw + lay.wa), *sA = sW + n1;
    uint8_t *sK = smem_raw + lay.sk, *sLvl = smem_raw + lay.lvl;      // [depth - 1][type][length]: level of the stage, 255: does not fit
    Bits<W> *sOk = reinterpret_cast<Bits<W> *>(smem_raw + lay.a);     // [depth & 1][type][length][same-type link][type before]
    Bits<W> *sReach = reinterpret_cast<Bits<W> *>(smem_raw + lay.reach);
    u32 *sM = reinterpret_cast<u32 *>(smem_raw + lay.m);              // [type][length][level][transfer][word]: bit k: (k, k + n] costs at most B
    longlong2 *sSpan = reinterpret_cast<longlong2 *>(smem_raw + lay.span);    // [type][length][level]: least and most that n layers cost
    i64 *sLeast = reinterpret_cast<i64 *>(smem_raw + lay.least);              // ... least, first and last stages included
    i64 *sMean = reinterpret_cast<i64 *>(smem_raw + lay.mean);                // ... mean
    u32 *sFin = reinterpret_cast<u32 *>(smem_raw + lay.fin);          // [type][length]: transfers under which the last stage costs at most B
    dp_prologue_rows<i64, LINEAR>(dc, p, c2, coef, coef, true, T, RW, 0xffffffffu, nwarps, sR, sW, sA, sK, minfo, sP2P, szero);
    for (int e = tid; e < 2 * HAP_MAX_TYPES * lmax; e += kReachThreads)             // (types that do not exist stay empty)
#pragma unroll
        for (int w = 0; w < W; ++w) sReach[e].w[w] = 0;
    const i64 *cfp = coef + (size_t)p * T * HAP_NCOEF;
    const i64 mx = cfp[HAP_MX], mpre = cfp[HAP_MPRE], mpost = cfp[HAP_MPOST];

    auto cost = [&](int t, int r, int k, int j) -> i64 {
        const i64 *rM = sR + (size_t)t * RW * n1;
        if (LINEAR) return rM[(size_t)r * n1 + j] - rM[(size_t)r * n1 + k];
        return (rM[j] - rM[k]) + tau_term((i64)dc.tau_q[r], rM[n1 + j] - rM[n1 + k]);
    };
    for (int g = wib; g < T * nwin * R; g += nwarps) {
        const int r = g % R, q = (g / R) % nwin, t = g / (R * nwin), n = jc.nmin[t] + q;
        i64 a = kInf, b = -1, any = kInf, sum = 0;            // of the stages between the first and the last; of all
        for (int k = lane; k + n <= N; k += 32) {
            const i64 c = cost(t, r, k, k + n);
            any = c < any ? c : any;
            sum += c;
            if (k > 0 && k + n < N) { a = c < a ? c : a; b = c > b ? c : b; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const i64 x = __shfl_xor_sync(0xffffffffu, a, o), y = __shfl_xor_sync(0xffffffffu, b, o);
            a = x < a ? x : a; b = y > b ? y : b;
            const i64 z = __shfl_xor_sync(0xffffffffu, any, o);
            any = z < any ? z : any;
        }
        sum = warp_sum_i64(sum);
        if (lane == 0) { sSpan[g] = make_longlong2(a, b); sLeast[g] = any; sMean[g] = n <= N ? sum / (N - n + 1) : kInf; }
    }
    __syncthreads();
    if (tid <= PP)
#pragma unroll
        for (int w = 0; w < W; ++w) { const int n = jc.width[tid] - 64 * w; s_level[tid].w[w] = n >= 64 ? ~0ull : n > 0 ? (1ull << n) - 1ull : 0ull; }
    // least and most of the transfers into a stage of a type 
    i64 *sK2 = &s_k2[0][0];
    if (tid < T) {                                            // (a type on its own with one stage has none)
        u32 via = 0;
        for (int h = 0; h < T; ++h) if (h != tid && jc.cnt[h] > 0) via |= 4u << h;
        for (int q = 1; q < jc.cnt[tid]; ++q) {
            const i64 first = (i64)q * pc.G;
            via |= (first - 1) / dc.node_size[tid] == first / dc.node_size[tid] ? 1u : 2u;
        }
        s_via[tid] = via;
        i64 a = kInf, b = 0;
        for (int e = 0; e < kReachKc; ++e)
            if ((via >> e) & 1u) { const i64 v = sP2P[tid][e]; a = v < a ? v : a; b = v > b ? v : b; }
        sK2[2 * tid] = a; sK2[2 * tid + 1] = b;
        const i64 pre = minfo[(1 << tid) - 1].kpre;
        s_kmin[tid] = pre < a ? pre : a;
    }
    __syncthreads();

    for (int pos = 0; pos < dc.n_rc; ++pos) {
        const int rc_idx = dc.rc_order[pos];
        const unsigned rc_mask = dc.rc_masks[rc_idx];
        // the answer under an earlier policy that allows more is a lower bound (kInf: infeasible here, too)
        i64 floor_b = 0;
        for (int q = 0; q < pos; ++q)
            if ((dc.rc_sup[pos] >> q) & 1u) { const i64 v = s_res[q]; floor_b = v > floor_b ? v : floor_b; }
        i64 result = kInf;
        if (floor_b < kInf) {
            // ---- recomputation level of a stage of n layers at each depth and type ---------------------------------
            if (tid < HAP_MAX_TYPES) s_used[tid] = 0;
            __syncthreads();
            for (int e = tid; e < PP * T * nwin; e += kReachThreads) {
                const int q = e % nwin, t = (e / nwin) % T, i = e / (nwin * T) + 1, n = jc.nmin[t] + q;
                int lv = 255;
                if (n <= jc.nmax[t] && n <= N) {
                    const i64 extra = (i == 1 ? mpre : 0) + (i == PP ? mpost : 0);
                    const int inflight = PP - i + 1;
                    const i64 mstore = pc.M < inflight ? pc.M : inflight, cap = dc.cap_eff[t];
                    // behind the first stage every span is of one layer kind, so its last possible place stands for all
                    const int k = i == 1 ? 0 : N - n;
                    for (int r = R - 1; r >= 0; --r)
                        if (((rc_mask >> r) & 1u) && span_fits(sW, sA, sK, extra, mx, mstore, cap, (i64)dc.xi_q[r], k, k + n)) lv = r;
                }
                sLvl[e] = (uint8_t)lv;
                if (lv != 255 && i > 1 && i < PP && !((s_used[t] >> lv) & 1u)) atomicOr(&s_used[t], 1u << lv);
            }
            if (PP == 1) {
                __syncthreads();
                // one stage of all layers
                for (int t = 0; t < T; ++t)
                    if (jc.cnt[t] > 0 && jc.nmin[t] <= N && N <= jc.nmax[t]) {
                        const int lv = sLvl[t * nwin + N - jc.nmin[t]];
                        if (lv != 255) { const i64 v = cost(t, lv, 0, N) + minfo[(1 << t) - 1].kpre + minfo[(1 << t) - 1].kpost; result = v < result ? v : result; }
                    }
            } else {
                // whether no stage has to cost more than B; the answer is then at most s_dn <= B, else at least s_up > B
                auto test = [&](i64 B) -> bool {
                    __syncthreads();
                    if (tid == 0) { s_dn = 0; s_up = (u64)kInf; }
                    __syncthreads();
                    i64 dn = 0, up = kInf;
                    u32 near_dn = 0, near_up = ~0u;          // costs within 2^32 ns of B, as cost - (B + 1)
                    auto see = [&](i64 v) { if (v <= B) dn = v > dn ? v : dn; else up = v < up ? v : up; return v <= B; };
                    for (int g = wib; g < T * nwin * R; g += nwarps) {
                        const int r = g % R, q = (g / R) % nwin, t = g / (R * nwin), n = jc.nmin[t] + q;
                        if (!((s_used[t] >> r) & 1u) || n > jc.nmax[t] || jc.cnt[t] == 0) continue;
                        const longlong2 range = sSpan[g];
                        if (range.y < 0) {                                    // no room between a first and a last stage
                            for (int e = lane; e < kReachKc * mw; e += 32) sM[(size_t)g * kReachKc * mw + e] = 0u;
                            continue;
                        }
                        const i64 least = range.x + s_k2[t][0], most = range.y + s_k2[t][1];
                        if (most <= B || least > B) {
                            // all of them or none: most lengths, once B is near the answer
                            see(most <= B ? most : least);
                            for (int e = lane; e < kReachKc * mw; e += 32) {
                                const int f = e / mw, w = e - f * mw;
                                // bits 1 .. N - n - 1
                                const int top = N - n - w * 32;
                                u32 v = most > B || !((s_via[t] >> f) & 1u) || top <= 0 ? 0u : top >= 32 ? ~0u : (1u << top) - 1u;
                                if (w == 0) v &= ~1u;
                                sM[(size_t)g * kReachKc * mw + e] = v;
                            }
                            continue;
                        }
                        see(B + 1 - 4294967296ll);                            // (costs further away than that are not looked at)
                        up = B + 4294967296ll < up ? B + 4294967296ll : up;
                        const u32 via = s_via[t];
                        for (int w = 0; w < mw; ++w) {
                            const int k = w * 32 + lane;
                            const bool in = k >= 1 && k + n < N;              // a stage that is neither the first nor the last
                            const i64 c = (in ? cost(t, r, k, k + n) : kInf) - (B + 1);       // (negative: at most B)
                            u32 mine = 0;
#pragma unroll
                            for (int e = 0; e < kReachKc; ++e) {
                                if (!((via >> e) & 1u)) continue;
                                const i64 x = c + sP2P[t][e];
                                const int hi = (int)(x >> 32);
                                const u32 lw = (u32)x;
                                if (hi == -1) near_dn = lw > near_dn ? lw : near_dn;
                                if (hi == 0) near_up = lw < near_up ? lw : near_up;
                                const u32 b = __ballot_sync(0xffffffffu, hi < 0);
                                if (lane == e) mine = b;
                            }
                            if (lane < kReachKc) sM[((size_t)(g * kReachKc + lane)) * mw + w] = mine;
                        }
                    }
                    // first and last stages: one length each
                    for (int e = tid; e < T * nwin; e += kReachThreads) {
                        const int q = e % nwin, t = e / nwin, n = jc.nmin[t] + q;
                        u32 okl = 0;
                        if (n <= jc.nmax[t] && n < N && jc.cnt[t] > 0) {
                            const int lv = sLvl[((size_t)(PP - 1) * T + t) * nwin + q];
                            if (lv != 255) {
                                const i64 c = cost(t, lv, N - n, N) + minfo[(1 << t) - 1].kpost;
                                for (int f = 0; f < 2 + T; ++f)
                                    if (((s_via[t] >> f) & 1u) && see(c + sP2P[t][f])) okl |= 1u << f;
                            }
                            const int l1 = sLvl[(size_t)t * nwin + q];
                            if (l1 != 255 && see(cost(t, l1, 0, n) + minfo[(1 << t) - 1].kpre)) okl |= 1u << 16;
                        }
                        sFin[e] = okl;
                    }
                    near_dn = __reduce_max_sync(0xffffffffu, near_dn); near_up = __reduce_min_sync(0xffffffffu, near_up);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const i64 a = __shfl_xor_sync(0xffffffffu, dn, o), b = __shfl_xor_sync(0xffffffffu, up, o);
                        dn = a > dn ? a : dn; up = b < up ? b : up;
                    }
                    if (near_dn) { const i64 v = (B + 1) - 4294967296ll + (i64)near_dn; dn = v > dn ? v : dn; }
                    if (near_up != ~0u) { const i64 v = (B + 1) + (i64)near_up; up = v < up ? v : up; }
                    if (lane == 0) { atomicMax(&s_dn, (u64)dn); atomicMin(&s_up, (u64)up); }
                    __syncthreads();
                    // masks of a depth: the words of the level that its memory allows, from the first end layer of the level before
                    auto masks_of = [&](int i, int turn) {
                        const int at = jc.base[i - 1], w0 = at >> 5, s = at & 31;
                        const Bits<W> all = s_level[i - 1];
                        const int per_t = (nwin * kReachOk + 31) & ~31;
                        for (int e0 = wib * 32; e0 < T * per_t; e0 += kReachThreads) {          // (a warp stays inside one type)
                            const int t = e0 / per_t, e = e0 - t * per_t + lane;
                            const int h = e & (HAP_MAX_TYPES - 1), f = h == t ? (e / HAP_MAX_TYPES) & 1 : 2 + h, q = e / kReachOk;
                            Bits<W> b;
#pragma unroll
                            for (int w = 0; w < W; ++w) b.w[w] = 0;
                            const bool in = q < nwin, there = in && jc.cnt[t] > 0 && ((s_via[t] >> f) & 1u);
                            const int lv = there ? sLvl[((size_t)(i - 1) * T + t) * nwin + q] : 255;
                            if (lv != 255) {
                                const u32 *m = sM + ((size_t)((t * nwin + q) * R + lv) * kReachKc + f) * mw;
                                u32 v[2 * W + 1];
#pragma unroll
                                for (int w = 0; w <= 2 * W; ++w) v[w] = w0 + w < mw ? m[w0 + w] : 0u;
#pragma unroll
                                for (int w = 0; w < W; ++w)
                                    b.w[w] = (u64)__funnelshift_r(v[2 * w], v[2 * w + 1], s) | (u64)__funnelshift_r(v[2 * w + 1], v[2 * w + 2], s) << 32;
                            }
                            bool full = true, empty = true;
#pragma unroll
                            for (int w = 0; w < W; ++w) { full = full && (b.w[w] & all.w[w]) == all.w[w]; empty = empty && b.w[w] == 0; }
                            const u32 not_full = __ballot_sync(0xffffffffu, there && !full), some = __ballot_sync(0xffffffffu, !empty);
                            if (in) {
                                sOk[(size_t)((i & 1) * T + t) * nwin * kReachOk + e] = b;
                                if ((lane & (kReachOk - 1)) == 0) {
                                    if ((some >> lane) & 0xffu) atomicMax(&s_end[turn][t], q + 1);
                                    if ((not_full >> lane) & 0xffu) atomicMin(&s_full[turn][t], q);
                                }
                            }
                        }
                    };
                    if (tid < 3 * HAP_MAX_TYPES) { s_end[tid / HAP_MAX_TYPES][tid % HAP_MAX_TYPES] = 0; s_full[tid / HAP_MAX_TYPES][tid % HAP_MAX_TYPES] = nwin; }
                    __syncthreads();
                    if (PP > 2) masks_of(2, 2);
                    // level 1
                    for (unsigned e = (unsigned)tid; e < jc.n_states[1] * (unsigned)T; e += kReachThreads) {
                        const unsigned t = e / jc.n_states[1], sl = e - t * jc.n_states[1];
                        Bits<W> b;
#pragma unroll
                        for (int w = 0; w < W; ++w) b.w[w] = 0;
                        if (jc.cnt[t] > 0 && sl == jc.first[t])
                            for (int q = 0; q < nwin; ++q)
                                if (sFin[t * nwin + q] >> 16) {
                                    const int bit = jc.nmin[t] + q - jc.base[1];
                                    if (bit >= 0 && bit < jc.width[1]) b.w[W == 1 ? 0 : bit >> 6] |= 1ull << (bit & 63);
                                }
                        sReach[(size_t)t * lmax + sl] = b;
                    }
                    __syncthreads();
                    for (int i = 2, turn = 2; i < PP; ++i, turn = turn == 2 ? 0 : turn + 1) {       // turn: i % 3
                        const Bits<W> *prv = sReach + (size_t)(i & 1 ? HAP_MAX_TYPES * lmax : 0);          // level 1 lies in the first buffer
                        Bits<W> *cur = sReach + (size_t)(i & 1 ? 0 : HAP_MAX_TYPES * lmax);
                        const unsigned ns = jc.n_states[i], total = ns * (unsigned)T;
                        const unsigned *ent = jc.ent + jc.ent_off[i];
                        const int d = jc.base[i] - jc.base[i - 1];
                        const Bits<W> *okd = sOk + (size_t)(i & 1) * T * nwin * kReachOk;
                        const Bits<W> lm = s_level[i];
                        const int turn_next = turn == 2 ? 0 : turn + 1, turn_free = 3 - turn - turn_next;
                        if (i + 1 < PP) masks_of(i + 1, turn_next);
                        if (tid < HAP_MAX_TYPES) { s_end[turn_free][tid] = 0; s_full[turn_free][tid] = nwin; }
                        int some = 0;
                        // lengths are gathered by Horner's rule from the longest on, one position a step; a bit that leaves the words at
                        // the top lies outside the level (joint_reach_class); those before nf are all alike
                        auto step_up = [&](Bits<W> &acc, const Bits<W> &x) {
#pragma unroll
                            for (int w = W - 1; w > 0; --w) acc.w[w] = acc.w[w] << 1 | acc.w[w - 1] >> 63 | x.w[w];
                            acc.w[0] = acc.w[0] << 1 | x.w[0];
                        };
                        for (unsigned e = (unsigned)tid; e < total; e += kReachThreads) {
                            const unsigned en = __ldg(ent + e), up_sl = en & 0xffffu;
                            const int t = (int)(en >> 16) & 3, cls = (int)(en >> 18) & 1;
                            Bits<W> acc;
#pragma unroll
                            for (int w = 0; w < W; ++w) acc.w[w] = 0;
                            if ((en >> 19) & 1u) {
                                if (!HAP_CHECK_OK(4, up_sl < jc.n_states[i - 1])) continue;
                                Bits<W> from[HAP_MAX_TYPES], any;
#pragma unroll
                                for (int h = 0; h < HAP_MAX_TYPES; ++h) from[h] = prv[(size_t)h * lmax + up_sl];
                                bool none = true;
#pragma unroll
                                for (int w = 0; w < W; ++w) {
                                    any.w[w] = from[0].w[w] | from[1].w[w] | from[2].w[w] | from[3].w[w];
                                    none = none && any.w[w] == 0;
                                }
                                if (!none) {
                                    const Bits<W> *ok = okd + (size_t)t * nwin * kReachOk + cls * HAP_MAX_TYPES;
                                    const int nf = s_full[turn][t];
                                    int q = s_end[turn][t] - 1;
                                    for (; q >= nf; --q) {
                                        const Bits<W> *o = ok + q * kReachOk;
                                        Bits<W> x;
#pragma unroll
                                        for (int w = 0; w < W; ++w)
                                            x.w[w] = (from[0].w[w] & o[0].w[w]) | (from[1].w[w] & o[1].w[w]) | (from[2].w[w] & o[2].w[w]) | (from[3].w[w] & o[3].w[w]);
                                        step_up(acc, x);
                                    }
                                    for (; q >= 0; --q) step_up(acc, any);
                                    acc = bits_shift<W>(acc, jc.nmin[t] - d);
#pragma unroll
                                    for (int w = 0; w < W; ++w) { acc.w[w] &= lm.w[w]; some |= acc.w[w] != 0; }
                                }
                            }
                            cur[(size_t)t * lmax + (e - (unsigned)t * ns)] = acc;
                        }
                        if (!__syncthreads_or(some)) return false;
                    }
                    // last stage
                    const Bits<W> *prv = sReach + (size_t)(PP & 1 ? HAP_MAX_TYPES * lmax : 0);
                    int done = 0;
                    for (int e = tid; e < T * nwin * T; e += kReachThreads) {
                        const int h = e % T, q = (e / T) % nwin, t = e / (T * nwin), n = jc.nmin[t] + q, bit = N - n - jc.base[PP - 1];
                        const u32 okl = sFin[t * nwin + q];
                        if (!(okl & 0xffffu) || bit < 0 || bit >= 64 * W) continue;
                        const int first = (jc.cnt[t] - 1) * pc.G;
                        const int f = h == t ? ((first - 1) / dc.node_size[t] == first / dc.node_size[t] ? 0 : 1) : 2 + h;
                        if (!((okl >> f) & 1u)) continue;
                        const Bits<W> b = prv[(size_t)h * lmax + jc.fin[t]];
                        done |= (int)((b.w[W == 1 ? 0 : bit >> 6] >> (bit & 63)) & 1ull);
                    }
                    return __syncthreads_or(done) != 0;
                };
                // The longest stages that cost at most B, at the level that the depth's memory asks for, have to add up to N, with the best
                // type at every depth and with the best depth for every type.  With the least cost of a length anywhere, that is a lower
                // bound on the answer -- where even the largest does not do, nothing is feasible --; with its mean cost, a guess at it.
                // The sums grow with B in steps at those costs; a warp per trial, eight a round.  Where the largest B leaves less than a tenth of
                // the layers to spare, whether anything is feasible is in doubt: of the configurations of 32, 256 and 1,024 devices that pass the bound,
                // 95 % of the infeasible ones lie there and 3 % of the others.  Asked first there instead of after three tests: 256 devices, 220
                // layers, nothing feasible 527 -> 283 us, 1,024 devices 2,201 -> 2,158; 1,024 devices, 255 layers (ten of 6,228 feasible) 2,174 -> 2,368.
                auto capacity = [&](const i64 *costs) -> i64 {
                    i64 a, b;                                         // a smallest and largest cost that may be the one
                    auto around = [&](i64 B, i64 &below, i64 &above) {       // the largest cost at most B, the smallest above
                        below = 0; above = kInf;
                        for (int t = 0; t < T; ++t)
                            for (int e = lane; jc.cnt[t] > 0 && e < nwin * R; e += 32) {
                                const i64 v = costs[t * nwin * R + e] + s_kmin[t];
                                if (v <= B) below = v > below ? v : below; else above = v < above ? v : above;
                            }
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) {
                            const i64 x = __shfl_xor_sync(0xffffffffu, below, o), y = __shfl_xor_sync(0xffffffffu, above, o);
                            below = x > below ? x : below; above = y < above ? y : above;
                        }
                    };
                    i64 x, y;
                    around(kInf - 1, b, y);
                    around(-1, x, a);
                    bool first = true;
                    while (first || a < b) {
                        // trials at (b - a) (1 .. 8) / 8 behind a: the last one is b
                        const i64 step = (b - a) / nwarps, m = wib == nwarps - 1 ? b : a + step * (wib + 1);
                        int best = 0, sum = 0;
                        for (int h = 0; h < T; ++h) {
                            int most = 0;
                            if (jc.cnt[h] > 0 && lane < PP) {
                                const uint8_t *lv = sLvl + ((size_t)lane * T + h) * nwin;
                                const i64 *c = costs + (size_t)h * nwin * R, limit = m - s_kmin[h];
                                for (int q = jc.nmax[h] - jc.nmin[h]; q >= 0; --q)
                                    if (lv[q] != 255 && c[q * R + lv[q]] <= limit) { most = jc.nmin[h] + q; break; }
                            }
                            best = most > best ? most : best;
                            sum += jc.cnt[h] * (int)__reduce_max_sync(0xffffffffu, (unsigned)most);
                        }
                        const int by_depth = (int)__reduce_add_sync(0xffffffffu, (unsigned)best);
                        const bool enough = sum >= N && by_depth >= N && !__any_sync(0xffffffffu, lane < PP && best == 0);
                        if (lane == 0) s_enough[wib] = enough;
                        if (first && lane == 0 && wib == nwarps - 1) s_spare = (sum < by_depth ? sum : by_depth) - N;
                        __syncthreads();
                        int k = 0;
                        while (k < nwarps && !s_enough[k]) ++k;
                        __syncthreads();
                        if (k == nwarps) return kInf;                 // (the first round's last trial is the largest cost)
                        first = false;
                        const i64 lo = a + step * k, hi = k == nwarps - 1 ? b : a + step * (k + 1);      // not enough at lo (k > 0), enough at hi
                        around(hi, b, y);
                        if (k > 0) { around(lo, x, y); a = y; }
                        else if (step == 0) b = a;
                    }
                    return b;
                };
                __syncthreads();                                      // (the levels of the stages)
                const i64 low = capacity(sLeast), guess = low < kInf ? capacity(sMean) : kInf;
                // (one place calls the test: it is long)
                if (low < kInf) {
                    LimitSearch search;
                    search.begin(low, floor_b, guess, s_spare * 10 < N);
                    while (true) {
                        const bool can = test(search.B);
                        if (!search.next(can, (i64)s_dn, (i64)s_up)) break;
                    }
                    result = search.lo;
                }
            }
        }
        if (tid == 0) { s_res[pos] = result; out[(size_t)p * dc.n_rc + rc_idx] = result; }
        __syncthreads();
    }
}

}  // namespace hap
