// Checks the task lists of the prefix trees of a cluster (test_tree_tasks.py; no GPU is needed): prints, per PP class, stages,
// iterations of 1, 2 and 4 end layers, parts, memory allocations of the build, and the faults found.  Arguments: layers, first MoE
// layer, window delta, nodes per type, node size.
#include "../paper_2609_39350_b200/csrc/hap_tree_host.h"

#include <cstdio>
#include <cstdlib>
#include <map>

using namespace hap;

static long allocations;
#ifndef __CUDA_ARCH__
void *operator new(size_t n) { ++allocations; return malloc(n); }
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
#endif

int main(int argc, char **argv)
{
    if (argc != 6) return 2;
    const i64 P[4] = {400000, 300000, 250000, 150000}, cap[4] = {80ll << 30, 64ll << 30, 48ll << 30, 32ll << 30};
    DevConst dc{};
    dc.N = atoi(argv[1]); dc.kind_uniform_from = atoi(argv[2]);
    dc.delta_q = atoi(argv[3]); dc.R = 2; dc.tau_linear = 1;
    i64 W = 0;
    for (char *s = strtok(argv[4], ","); s && dc.T < HAP_MAX_TYPES; s = strtok(nullptr, ",")) {
        const int h = dc.T++;
        dc.node_size[h] = atoi(argv[5]); dc.m[h] = (i64)atoi(s) * dc.node_size[h]; dc.P[h] = P[h]; dc.cap_eff[h] = cap[h];
        W += dc.m[h];
    }
    for (int PP = 1; PP <= HAP_MAX_PP && PP <= dc.N; PP *= 2) {
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
        in.dc = &dc; in.rep = q; in.n_conf = 1000; in.n_sm = 148; in.want_tree = true;
        TreeClassHost th;
        allocations = 0;
        TreeBuilder(in).build(th);
        const long allocated = allocations;
        if (!th.ok) return 3;
        const TreeClass &c = th.cls;
        long iters[5] = {0, 0, 0, 0, 0}, faults = 0;
        double work = 0, chain = 0;                                                  // instructions, from the tasks as they are laid out
        for (const TreePartHost &ph : th.parts) {
            u32 e = 0, behind_choices = 0;
            double part = (double)((ph.meta.nmap + 31) / 32) * (kTreeLeaf + kTreePerStage * PP);
            for (u32 q = 0; q < 32 * ph.meta.n_iter; q += 32) {
                int most = 1;
                for (u32 i = q; i < q + 32; ++i)
                    if (ph.tasks[i].y >> 24 & 7u) most = std::max(most, (int)(ph.tasks[i].y >> 16 & 255u) - (int)(ph.tasks[i].y >> 8 & 255u) + 1);
                const u32 J = ph.tasks[q].w >> 16 & 7u;
                part += kTreeIteration[J / 2] + kTreePerLength[J / 2] * most;
            }
            work += part; chain = std::max(chain, part);
            faults += ph.tasks.size() != 32u * (ph.meta.n_iter + 1);                  // the iteration behind the last is there to be asked for
            for (u32 q = 32 * ph.meta.n_iter; q < ph.tasks.size(); ++q) faults += (ph.tasks[q].y >> 24 & 7u) != 0 || (ph.tasks[q].y >> 8 & 255u) <= (ph.tasks[q].y >> 16 & 255u);
            for (int d = 1; d < PP; ++d) {
                // every row (a run of slots between padding) is covered slot by slot, once; its first task writes the padding in
                // front, one task of the depth that behind the last row
                std::map<u32, u32> cover;
                std::vector<u32> first;
                int last = 0;
                u32 top = 0;
                u32 first_choice = ~0u, last_choice = 0;
                bool ends = false;
                for (; !ends || e % 32; ++e) {
                    if (e >= 32 * ph.meta.n_iter) { ++faults; break; }
                    const TreeTask &t = ph.tasks[e];
                    const u32 cnt = t.y >> 24 & 7u, slot = t.x >> 16, J = t.w >> 16 & 7u;
                    ends = t.w & kTaskEnds;
                    if (e % 32 == 0) ++iters[J];
                    else faults += t.w >> 16 != ph.tasks[e - 1].w >> 16;            // alike in an iteration
                    faults += !(J == 1 || J == 2 || J == 4) || cnt > J || (t.w >> 20 & 1u) != !c.flat[d] || (!c.flat[d] && J != 1);
                    if (cnt == 0) { faults += (t.y >> 27 & 3u) || (t.y >> 8 & 255u) <= (t.y >> 16 & 255u); continue; }      // fills up
                    faults += (t.z >> 16) / HAP_MAX_TYPES != (u32)d - 1;
                    first_choice = std::min(first_choice, (t.w & 0xffffu) - slot); last_choice = std::max(last_choice, (t.w & 0xffffu) + cnt);
                    faults += (t.w & 0xffffu) - slot != first_choice || (t.w & 0xffffu) < behind_choices || (t.w & 0xffffu) + cnt > c.ch_bytes;
                    for (u32 i = 0; i < cnt; ++i) faults += ++cover[slot + i] != 1 || slot + i >= c.buf_cells[d & 1];
                    if (t.y >> 27 & 1u) first.push_back(slot);
                    if (t.y >> 28 & 1u) { ++last; top = slot + cnt; }
                }
                behind_choices = last_choice;
                size_t runs = 0;
                u32 behind = 0;
                for (const auto &[s, n] : cover) {
                    if (s != behind) { ++runs; faults += std::find(first.begin(), first.end(), s) == first.end() || (runs > 1 && s - behind != kTreePad); }
                    behind = s + 1;
                }
                faults += first.size() != runs || (runs && (last != 1 || top != behind)) || behind + kTreePad > c.buf_cells[d & 1] + (runs ? 0 : kTreePad);
            }
            faults += e != 32 * ph.meta.n_iter;
        }
        // the estimate that the parts were chosen by (an iteration whose tasks all came out narrower than planned takes less)
        faults += work > th.work || work < 0.95 * th.work || chain > th.chain || chain < 0.95 * th.chain;
        printf("%d %ld %ld %ld %zu %ld %ld\n", PP, iters[1], iters[2], iters[4], th.parts.size(), allocated, faults);
    }
    return 0;
}
