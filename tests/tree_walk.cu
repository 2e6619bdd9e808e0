// Walks the prefix trees of a cluster on the host, task by task as tree_dp_kernel does, with stage costs of its own, and compares every
// mapping's bottleneck and partition with a recurrence over that mapping alone (test_tree_tasks.py; no GPU is needed).  Prints,
// per PP class, stages, mappings, and the faults found.  Arguments: layers, first MoE layer, window delta, nodes per type, node
// size, configurations a class.
#include "../paper_2609_39350_b200/csrc/hap_tree_host.h"

#include <cstdio>
#include <cstdlib>
#include <random>

using namespace hap;

int main(int argc, char **argv)
{
    if (argc != 7) return 2;
    const i64 P[4] = {400000, 300000, 250000, 150000}, cap[4] = {80ll << 30, 64ll << 30, 48ll << 30, 32ll << 30};
    DevConst dc{};
    const int N = dc.N = atoi(argv[1]);
    dc.kind_uniform_from = atoi(argv[2]); dc.delta_q = atoi(argv[3]); dc.R = 2; dc.tau_linear = 1;
    i64 W = 0;
    for (char *s = strtok(argv[4], ","); s && dc.T < HAP_MAX_TYPES; s = strtok(nullptr, ",")) {
        const int h = dc.T++;
        dc.node_size[h] = atoi(argv[5]); dc.m[h] = (i64)atoi(s) * dc.node_size[h]; dc.P[h] = P[h]; dc.cap_eff[h] = cap[h];
        W += dc.m[h];
    }
    std::mt19937 rng(N);
    const double inf = 1e300, poison = -1.0;                    // (poison: an entry that no task wrote would win every comparison)
    for (int PP = 1; PP <= HAP_MAX_PP && PP <= N; PP *= 2) {
        if (W % PP) continue;
        hap_pconf q{};
        q.PP = PP; q.G = (int)(W / PP); q.mode = HAP_MAP_MULTISET; q.nmap = 1;
        int placed = 0;
        for (int h = 0; h < dc.T; ++h) {
            if (dc.m[h] % q.G) q.mode = HAP_MAP_BLOCK;
            for (int c = 1; c <= dc.m[h] / q.G && q.nmap < (1u << 20); ++c) q.nmap = q.nmap * (u64)++placed / (u64)c;
        }
        if (q.nmap > 2048) q.mode = HAP_MAP_BLOCK;
        if (q.mode == HAP_MAP_BLOCK) { q.nmap = 1; for (int h = 2; h <= dc.T; ++h) q.nmap *= (u64)h; }
        TreeInputs in{};
        in.dc = &dc; in.rep = q; in.n_conf = (size_t)atoi(argv[6]); in.n_sm = 148; in.want_tree = true;
        TreeClassHost th;
        TreeBuilder(in).build(th);
        if (!th.ok) return 3;
        const TreeClass &c = th.cls;
        // stage costs: a constant per first type or transfer, and prefix sums per row group (few values, so that many are equal)
        std::vector<double> K(kTreeKtab), row((size_t)c.n_mrows * (N + 1));
        for (double &v : K) v = rng() % 4;
        for (int g = 0; g < c.n_mrows; ++g)
            for (int j = 1; j <= N; ++j) row[(size_t)g * (N + 1) + j] = row[(size_t)g * (N + 1) + j - 1] + 1 + rng() % 3;
        auto cost = [&](u32 k, u32 g, int j, int n) { return K[k] + row[(size_t)g * (N + 1) + j] - row[(size_t)g * (N + 1) + j - n]; };
        long faults = 0;
        for (const TreePartHost &ph : th.parts) {
            std::vector<double> buf[2], zero(kTreeAhead + 2 * kTreePad + 1, inf);
            std::vector<u32> choice(c.ch_bytes, 0);
            zero[kTreeAhead + kTreePad] = 0.0;
            for (int b = 0; b < 2; ++b) buf[b].assign(c.buf_cells[b], poison);
            // cells of a scan, from entry `src` of `prev` (which holds length a of cell 0) on
            auto scan = [&](const std::vector<double> &prev, long src, int j, int i, int a, int b, u32 k, u32 g, int &arg) {
                double best = inf;
                arg = 0;
                for (int n = a; n <= b; ++n) {
                    const long at = src + i - (n - a);
                    if (at < 0 || at >= (long)prev.size() || (j + i - n < 0 && prev[(size_t)at] < inf)) { ++faults; continue; }
                    if (j + i - n < 0) continue;                // (in front of the first layer: infinite whatever the row says)
                    const double v = std::max(prev[(size_t)at], cost(k, g, j + i, n));
                    if (v < inf && v <= best) { best = v; arg = n; }
                }
                return best;
            };
            u32 e = 0;
            for (int d = 1; d < PP; ++d) {
                const std::vector<double> &prev = d == 1 ? zero : buf[(d & 1) ^ 1];
                std::vector<double> &cur = buf[d & 1];
                std::fill(cur.begin(), cur.end(), poison);
                bool ends = false;
                for (; !ends || e % 32; ++e) {
                    if (e >= 32 * ph.meta.n_iter) { ++faults; break; }
                    const TreeTask &t = ph.tasks[e];
                    ends = t.w & kTaskEnds;
                    const int j = (int)(t.y & 255u), a = (int)(t.y >> 8 & 255u), b = (int)(t.y >> 16 & 255u), cnt = (int)(t.y >> 24 & 7u);
                    const long src = (long)(t.x & 0xffffu), dst = (long)(t.x >> 16);
                    // a scan asks for the two entries below its last one, and at its first length for as many as it is wide: those past the
                    // task's own cells, which nothing is taken from, may lie in the words behind the buffer
                    const long J = (long)(t.w >> 16 & 7u);
                    if (a <= b) faults += src - (b - a + 2) < 0 || src + cnt - 1 >= (long)prev.size() || src + J - 1 >= (long)(prev.size() + kTreeSmemFixed / 8);
                    for (int i = 0; i < cnt; ++i) {
                        int arg;
                        const double v = scan(prev, src, j, i, a, b, t.z & 255u, t.z >> 8 & 255u, arg);
                        cur[(size_t)(dst + i)] = arg ? v : inf; choice[(t.w & 0xffffu) + (u32)i] = (u32)arg;
                    }
                    if (t.y >> 27 & 1u) for (long i = 1; i <= kTreePad; ++i) cur[(size_t)(dst - i)] = inf;
                    if (t.y >> 28 & 1u) for (long i = 0; i < kTreePad; ++i) cur[(size_t)(dst + cnt + i)] = inf;
                }
            }
            const std::vector<double> &prev = PP == 1 ? zero : buf[(PP - 1) & 1];
            for (u32 m = 0; m < ph.meta.nmap; ++m) {
                // the mapping on its own: windows from the shares of its types' compute power, smallest split on ties
                i64 Ps = 0, Pm[HAP_MAX_PP];
                u32 mask[HAP_MAX_PP], kidx[HAP_MAX_PP];
                for (int s = 0; s < PP; ++s) {
                    const StageMap sm = decode_stage(dc, q, ph.meta.m_lo + m, s);
                    mask[s] = (u32)sm.mask; Pm[s] = 1ll << 60;
                    for (int h = 0; h < dc.T; ++h) if (sm.mask >> h & 1) Pm[s] = std::min(Pm[s], dc.P[h]);
                    Ps += Pm[s];
                    kidx[s] = s == 0 ? (u32)c.mrow_of[sm.mask] : (u32)(16 + sm.hb * 6 + (sm.cls == HAP_CROSS ? 2 + sm.ha : sm.cls));
                }
                std::vector<double> f(N + 1, inf);
                std::vector<std::vector<int>> cut(PP + 1, std::vector<int>(N + 1, 0));
                f[0] = 0.0;
                for (int d = 1; d <= PP; ++d) {
                    i64 lo = 1, hi = N - PP + 1;
                    if (dc.delta_q >= 0) {
                        lo = std::max<i64>(lo, (1024 - dc.delta_q) * Pm[d - 1] * N / (1024 * Ps));
                        hi = std::min<i64>(hi, ((1024 + dc.delta_q) * Pm[d - 1] * N + 1024 * Ps - 1) / (1024 * Ps));
                    }
                    std::vector<double> next(N + 1, inf);
                    for (int j = 1; j <= N; ++j)
                        for (int n = (int)lo; n <= (int)hi && n <= j; ++n) {
                            const double v = std::max(f[j - n], cost(kidx[d - 1], c.mrow_of[mask[d - 1]], j, n));
                            if (v < inf && v <= next[j]) { next[j] = v; cut[d][j] = n; }
                        }
                    f.swap(next);
                }
                const int a = (int)(ph.leaf[m] & 255u), b = (int)(ph.leaf[m] >> 8 & 255u);
                u32 pw = ph.path[(size_t)(PP - 1) * ph.meta.nmap + m];
                int n = 0;
                double v = inf;
                if (a <= b) {
                    const long src = (long)(pw & 0xfffffu);
                    faults += src - (b - a + 2) < 0 || src >= (long)prev.size();
                    v = scan(prev, src, N, 0, a, b, pw >> 20 & 63u, pw >> 26 & 15u, n);
                }
                faults += v != f[N];
                if (v == inf || f[N] == inf) continue;
                int j = N;
                for (int d = PP; d >= 1; --d) {
                    faults += n != cut[d][j] || (pw >> 20 & 63u) != kidx[d - 1] || (pw >> 26 & 15u) != c.mrow_of[mask[d - 1]];
                    j -= n;
                    if (d == 1 || n < 1 || j < 0) break;
                    pw = ph.path[(size_t)(d - 2) * ph.meta.nmap + m];
                    const long at = (long)(pw & 0xfffffu) - 256 + j;
                    n = at >= 0 && at < (long)choice.size() ? (int)choice[(size_t)at] : 0;
                }
                faults += j != 0;
            }
        }
        printf("%d %llu %ld\n", PP, (unsigned long long)q.nmap, faults);
    }
    return 0;
}
