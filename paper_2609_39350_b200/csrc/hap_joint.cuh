// Joint recurrence over the device-group state as a search for the bottleneck (sm_100a).
//
// The smallest bottleneck over all stage-type sequences of a configuration is the smallest B for which some sequence has a
// partition without a stage above B.  For a given B a state u (stages of each type placed) with last type t needs one bit
// per end layer instead of a value:
//     reach[u][t] = OR over stage lengths n, OR over types t' of the stage before,
//                   (reach[u - e_t][t'] AND ok[t][t'][n]) << n
// where bit k of ok says that layers (k, k + n] on type t cost at most B behind a stage of type t' and fit the memory of
// this depth.  All bits of a state sit in one or two 64-bit words (bits count from the smallest end layer of the level), so
// a level of every state takes a few logic instructions per (type, type before, length) and both levels of the recurrence
// stay in shared memory.  The stage costs are finitely many numbers: after a test, B moves to the nearest of them, so the
// bisection ends after about a dozen tests, each exact.
//
// One block per configuration.  Bound by instruction issue of the level loop: per (state, type) four logic operations per
// (type before, length).  The value form -- a 64-bit minimum per end layer and split, rows in
// global memory -- is kept for classes whose bits or masks do not fit (joint_dp_kernel).
#pragma once
#include "hap_device.cuh"

namespace hap {

constexpr int kReachThreads = 256;
constexpr int kReachKc = 2 + HAP_MAX_TYPES;       // transfer into a stage: same type intra / inter node, from type 0..3

struct JointReach {
    int PP, lmax, words;                          // stages; most states of a level; 64-bit words per state and type
    int nwin;                                     // most stage lengths of a type
    int nmin[HAP_MAX_TYPES], nmax[HAP_MAX_TYPES], cnt[HAP_MAX_TYPES];
    int fin[HAP_MAX_TYPES];                       // slot, at level PP - 1, of "one stage of type t left"
    unsigned id_lo, n_ids;                        // its configurations in the id list
    unsigned first[HAP_MAX_TYPES];                // slot, at level 1, of "one stage of type t placed"
    unsigned ent_off[HAP_MAX_PP + 1];             // level i's entries: [type][state] slot before | type << 16 | same-type link << 18 | valid << 19
    unsigned n_states[HAP_MAX_PP + 1];
    int base[HAP_MAX_PP + 1];                     // end layer of bit 0
    const unsigned *ent;
};

template <int W> struct Bits { u64 w[W]; };

template <int W>
__device__ __forceinline__ Bits<W> bits_shift(const Bits<W> &x, int s)      // by s towards higher end layers (s < 0: lower)
{
    Bits<W> y;
    if (W == 1) y.w[0] = s >= 0 ? (s < 64 ? x.w[0] << s : 0) : (s > -64 ? x.w[0] >> -s : 0);
    else {
        const u64 lo = x.w[0], hi = x.w[W - 1];
        if (s >= 0) {
            y.w[0] = s < 64 ? lo << s : 0;
            y.w[W - 1] = s == 0 ? hi : s < 64 ? (hi << s) | (lo >> (64 - s)) : s < 128 ? lo << (s - 64) : 0;
        } else {
            const int r = -s;
            y.w[W - 1] = r < 64 ? hi >> r : 0;
            y.w[0] = r < 64 ? (lo >> r) | (hi << (64 - r)) : r < 128 ? hi >> (r - 64) : 0;
        }
    }
    return y;
}

__host__ __device__ inline int reach_mask_words(int N) { return (N + 1 + 31) / 32; }

struct ReachSmem { u32 rows, wa, sk, m, a, reach, lvl, fin, total; };
__host__ __device__ inline ReachSmem reach_smem(int N, int T, int R, int RW, int PP, int lmax, int nwin, int words)
{
    auto up = [](size_t v) { return (u32)((v + 15) / 16 * 16); };
    const size_t n1 = (size_t)N + 1, depth = PP > 2 ? PP - 2 : 0;
    ReachSmem s;
    size_t o = 0;
    s.rows = (u32)o; o = up(o + (size_t)T * RW * n1 * 8);
    s.wa = (u32)o; o = up(o + 2 * n1 * 8);
    s.sk = (u32)o; o = up(o + n1);
    s.a = (u32)o; o = up(o + depth * T * nwin * kReachKc * words * 8);
    s.reach = (u32)o; o = up(o + (size_t)2 * T * lmax * words * 8);
    s.m = (u32)o; o = up(o + (size_t)T * nwin * R * kReachKc * reach_mask_words(N) * 4);
    s.fin = (u32)o; o = up(o + (size_t)T * nwin * 4);
    s.lvl = (u32)o; o = up(o + (size_t)PP * T * nwin);
    s.total = (u32)(o > 0xffffffffull ? 0xffffffffull : o);
    return s;
}

template <bool LINEAR, int W>
__global__ void __launch_bounds__(kReachThreads, 4)
joint_reach_kernel(const DevConst dc, const JointReach *classes, int n_classes, const unsigned *ids, const i64 *c2, const i64 *coef, i64 *out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ JointReach jc;
    __shared__ MaskInfo<i64> minfo[kMaxMasks];
    __shared__ i64 sP2P[HAP_MAX_TYPES][6];
    __shared__ i64 szero[1];
    __shared__ u64 s_dn, s_up;                              // largest stage cost that is at most B, smallest one above
    __shared__ double s_est;
    __shared__ i64 s_res[HAP_MAX_RC_MASKS];
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
    Bits<W> *sOk = reinterpret_cast<Bits<W> *>(smem_raw + lay.a);     // [depth - 2][type][length][transfer]
    Bits<W> *sReach = reinterpret_cast<Bits<W> *>(smem_raw + lay.reach);
    u32 *sM = reinterpret_cast<u32 *>(smem_raw + lay.m);              // [type][length][level][transfer][word]: bit k: (k, k + n] costs at most B
    u32 *sFin = reinterpret_cast<u32 *>(smem_raw + lay.fin);          // [type][length]: transfers under which the last stage costs at most B
    dp_prologue_rows<i64, LINEAR>(dc, p, c2, coef, coef, true, T, RW, 0xffffffffu, nwarps, sR, sW, sA, sK, minfo, sP2P, szero);
    const i64 *cfp = coef + (size_t)p * T * HAP_NCOEF;
    const i64 mx = cfp[HAP_MX], mpre = cfp[HAP_MPRE], mpost = cfp[HAP_MPOST];

    auto cost = [&](int t, int r, int k, int j) -> i64 {
        const i64 *rM = sR + (size_t)t * RW * n1;
        if (LINEAR) return rM[(size_t)r * n1 + j] - rM[(size_t)r * n1 + k];
        return (rM[j] - rM[k]) + tau_term((i64)dc.tau_q[r], rM[n1 + j] - rM[n1 + k]);
    };
    // lower bound on the bottleneck: with weights s_h, s_h B is at least the weighted time of a stage's layers on its type,
    // so B sum_stages s >= sum over layers of the smallest weighted time.  Weights: the types' speeds.
    if (wib == 0) {
        double s[HAP_MAX_TYPES], den = 0.0;
        for (int h = 0; h < T; ++h) { const i64 v = cost(h, 0, 0, N); s[h] = 1.0 / (double)(v > 0 ? v : 1); den += s[h] * (double)jc.cnt[h]; }
        double sum = 0.0;
        for (int l = lane; l < N; l += 32) {
            double m = 0.0;
            for (int h = 0; h < T; ++h) {
                const i64 *rM = sR + (size_t)h * RW * n1;
                i64 c = rM[l + 1] - rM[l];
                if (LINEAR) for (int r = 1; r < R; ++r) { const i64 x = rM[(size_t)r * n1 + l + 1] - rM[(size_t)r * n1 + l]; c = x < c ? x : c; }
                const double v = s[h] * (double)c;
                m = h == 0 || v < m ? v : m;
            }
            sum += m;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) s_est = sum / den * (1.0 - 1e-9);
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
                // whether no stage has to cost more than B; s_dn, s_up around B
                auto test = [&](i64 B) -> bool {
                    __syncthreads();
                    if (tid == 0) { s_dn = 0; s_up = (u64)kInf; }
                    __syncthreads();
                    i64 dn = 0, up = kInf;
                    auto see = [&](i64 v) { if (v <= B) dn = v > dn ? v : dn; else up = v < up ? v : up; return v <= B; };
                    for (int g = wib; g < T * nwin * R; g += nwarps) {
                        const int r = g % R, q = (g / R) % nwin, t = g / (R * nwin), n = jc.nmin[t] + q;
                        if (!((rc_mask >> r) & 1u) || n > jc.nmax[t] || jc.cnt[t] == 0) continue;
                        for (int w = 0; w < mw; ++w) {
                            const int k = w * 32 + lane;
                            const bool in = k >= 1 && k + n < N;              // a stage that is neither the first nor the last
                            const i64 c = in ? cost(t, r, k, k + n) : 0;
                            u32 mine = 0;
#pragma unroll
                            for (int e = 0; e < kReachKc; ++e) {
                                const int from = e < 2 ? t : e - 2;
                                if (from >= T || jc.cnt[from] == 0) continue;
                                bool ok = false;
                                if (in) ok = see(c + sP2P[t][e]);
                                const u32 b = __ballot_sync(0xffffffffu, ok);
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
                                    if (see(c + sP2P[t][f])) okl |= 1u << f;
                            }
                            const int l1 = sLvl[(size_t)t * nwin + q];
                            if (l1 != 255 && see(cost(t, l1, 0, n) + minfo[(1 << t) - 1].kpre)) okl |= 1u << 16;
                        }
                        sFin[e] = okl;
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const i64 a = __shfl_xor_sync(0xffffffffu, dn, o), b = __shfl_xor_sync(0xffffffffu, up, o);
                        dn = a > dn ? a : dn; up = b < up ? b : up;
                    }
                    if (lane == 0) { atomicMax(&s_dn, (u64)dn); atomicMin(&s_up, (u64)up); }
                    __syncthreads();
                    // masks of every depth: the words of the level that its memory allows, from the first end layer of the level before
                    for (int e = tid; e < (PP - 2) * T * nwin * kReachKc; e += kReachThreads) {
                        const int f = e % kReachKc, q = (e / kReachKc) % nwin, t = (e / (kReachKc * nwin)) % T, i = e / (kReachKc * nwin * T) + 2;
                        Bits<W> b;
#pragma unroll
                        for (int w = 0; w < W; ++w) b.w[w] = 0;
                        const int lv = sLvl[((size_t)(i - 1) * T + t) * nwin + q], from = f < 2 ? t : f - 2;
                        if (lv != 255 && jc.cnt[t] > 0 && from < T && jc.cnt[from] > 0) {
                            const u32 *m = sM + ((size_t)((t * nwin + q) * R + lv) * kReachKc + f) * mw;
                            const int at = jc.base[i - 1], w0 = at >> 5, s = at & 31;
                            u32 v[2 * W + 1];
#pragma unroll
                            for (int w = 0; w <= 2 * W; ++w) v[w] = w0 + w < mw ? m[w0 + w] : 0u;
#pragma unroll
                            for (int w = 0; w < W; ++w)
                                b.w[w] = (u64)__funnelshift_r(v[2 * w], v[2 * w + 1], s) | (u64)__funnelshift_r(v[2 * w + 1], v[2 * w + 2], s) << 32;
                        }
                        sOk[e] = b;
                    }
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
                                    if (bit >= 0 && bit < 64 * W) b.w[W == 1 ? 0 : bit >> 6] |= 1ull << (bit & 63);
                                }
                        sReach[(size_t)t * lmax + sl] = b;
                    }
                    __syncthreads();
                    for (int i = 2; i < PP; ++i) {
                        const Bits<W> *prv = sReach + (size_t)(i & 1 ? T * lmax : 0);          // level 1 lies in the first buffer
                        Bits<W> *cur = sReach + (size_t)(i & 1 ? 0 : T * lmax);
                        const unsigned ns = jc.n_states[i], total = ns * (unsigned)T;
                        const unsigned *ent = jc.ent + jc.ent_off[i];
                        const int d = jc.base[i] - jc.base[i - 1];
                        const Bits<W> *okd = sOk + (size_t)(i - 2) * T * nwin * kReachKc;
                        int some = 0;
                        for (unsigned e = (unsigned)tid; e < total; e += kReachThreads) {
                            const unsigned en = __ldg(ent + e), up_sl = en & 0xffffu;
                            const int t = (int)(en >> 16) & 3, cls = (int)(en >> 18) & 1;
                            Bits<W> acc;
#pragma unroll
                            for (int w = 0; w < W; ++w) acc.w[w] = 0;
                            if ((en >> 19) & 1u) {
                                if (!HAP_CHECK_OK(4, up_sl < jc.n_states[i - 1])) continue;
                                Bits<W> from[HAP_MAX_TYPES];
                                u64 any = 0;
#pragma unroll
                                for (int h = 0; h < HAP_MAX_TYPES; ++h) {
#pragma unroll
                                    for (int w = 0; w < W; ++w) from[h].w[w] = 0;
                                    if (h < T) from[h] = prv[(size_t)h * lmax + up_sl];
#pragma unroll
                                    for (int w = 0; w < W; ++w) any |= from[h].w[w];
                                }
                                if (any) {
                                    const Bits<W> *ok = okd + (size_t)t * nwin * kReachKc;
                                    const int lo = jc.nmin[t] - d, nl = jc.nmax[t] - jc.nmin[t] + 1;
                                    for (int q = 0; q < nl; ++q, ok += kReachKc) {
                                        Bits<W> x;
#pragma unroll
                                        for (int w = 0; w < W; ++w) x.w[w] = 0;
#pragma unroll
                                        for (int h = 0; h < HAP_MAX_TYPES; ++h)
                                            if (h < T) {
                                                const Bits<W> m = ok[h == t ? cls : 2 + h];
#pragma unroll
                                                for (int w = 0; w < W; ++w) x.w[w] |= from[h].w[w] & m.w[w];
                                            }
                                        x = bits_shift<W>(x, lo + q);
#pragma unroll
                                        for (int w = 0; w < W; ++w) acc.w[w] |= x.w[w];
                                    }
#pragma unroll
                                    for (int w = 0; w < W; ++w) some |= acc.w[w] != 0;
                                }
                            }
                            cur[(size_t)t * lmax + (e - (unsigned)t * ns)] = acc;
                        }
                        if (!__syncthreads_or(some)) return false;
                    }
                    // last stage
                    const Bits<W> *prv = sReach + (size_t)(PP & 1 ? T * lmax : 0);
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
                // between lo (no smaller stage cost can do) and hi (does): the next test lies above the lower bound by a
                // sixteenth first, then halfway
                __syncthreads();
                i64 lo = floor_b, hi;
                bool ok = true;
                if (floor_b > 0) ok = !test(floor_b);                // the larger choice of levels did not help: same answer
                if (!ok) result = floor_b;
                else {
                    if (floor_b > 0) lo = (i64)s_up;
                    if (test(kInf - 1)) {
                        hi = (i64)s_dn;
                        const i64 est = (i64)s_est;
                        if (est > lo) lo = est;
                        i64 step = lo / 16;
                        bool gallop = true;
                        while (lo < hi) {
                            i64 B = lo + (hi - lo) / 2;
                            if (gallop && step > 0 && lo + step < B) B = lo + step;
                            if (test(B)) { hi = (i64)s_dn; gallop = false; }
                            else { lo = (i64)s_up; step *= 2; }
                        }
                        result = hi;
                    }
                }
            }
        }
        if (tid == 0) { s_res[pos] = result; out[(size_t)p * dc.n_rc + rc_idx] = result; }
        __syncthreads();
    }
}

}  // namespace hap
