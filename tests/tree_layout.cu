// Prints what the host lays out for the prefix trees of a cluster, one line a PP class (test_tree_layout.py reads it; no
// GPU is needed).  Arguments: layers, first MoE layer, window delta, levels, nodes per type, node size, configurations a class.
#include "../paper_2609_39350_b200/csrc/hap_tree_host.h"

#include <cstdio>
#include <cstdlib>

using namespace hap;

int main(int argc, char **argv)
{
    if (argc != 8) return 2;
    const i64 P[4] = {400000, 300000, 250000, 150000}, cap[4] = {80ll << 30, 64ll << 30, 48ll << 30, 32ll << 30};
    DevConst dc{};
    dc.N = atoi(argv[1]); dc.kind_uniform_from = atoi(argv[2]);
    dc.delta_q = atoi(argv[3]); dc.R = atoi(argv[4]); dc.tau_linear = 1;
    i64 W = 0;
    for (char *s = strtok(argv[5], ","); s && dc.T < HAP_MAX_TYPES; s = strtok(nullptr, ",")) {
        const int h = dc.T++;
        dc.node_size[h] = atoi(argv[6]); dc.m[h] = (i64)atoi(s) * dc.node_size[h]; dc.P[h] = P[h]; dc.cap_eff[h] = cap[h];
        W += dc.m[h];
    }
    for (int PP = 1; PP <= HAP_MAX_PP && PP <= dc.N; PP *= 2) {
        if (W % PP) continue;
        hap_pconf q{};
        q.PP = PP; q.G = (int)(W / PP);
        bool homogeneous = true;
        u64 seqs = 1;
        int placed = 0;
        for (int h = 0; h < dc.T; ++h) {
            homogeneous = homogeneous && dc.m[h] % q.G == 0;
            for (int c = 1; c <= dc.m[h] / q.G && seqs < (1u << 20); ++c) seqs = seqs * (u64)++placed / (u64)c;
        }
        q.mode = homogeneous && seqs <= 2048 ? HAP_MAP_MULTISET : HAP_MAP_BLOCK;
        q.nmap = 1;
        for (int h = 2; h <= dc.T; ++h) q.nmap *= (u64)h;
        if (q.mode == HAP_MAP_MULTISET) q.nmap = seqs;
        TreeInputs in{};
        in.dc = &dc; in.rep = q; in.n_conf = (size_t)atoi(argv[7]); in.n_sm = 148; in.want_tree = true;
        TreeClassHost th;
        TreeBuilder(in).build(th);
        if (!th.ok) return 3;
        // entries of the row before that the scans read: the window of a task starts at its slot and moves down by one entry
        // a length, two further than the last (tree_scan asks for the next two before it knows that there are none)
        long low = 1 << 20;
        for (const TreePartHost &ph : th.parts) {
            for (const TreeTask &t : ph.tasks) {
                const long src = (long)(t.x & 0xffffu), a = t.y >> 8 & 255u, b = t.y >> 16 & 255u;
                if (a <= b) low = std::min(low, src - (b - a + 2));
            }
            for (u32 m = 0; m < ph.meta.nmap; ++m) {
                const long a = ph.leaf[m] & 255u, b = ph.leaf[m] >> 8 & 255u;
                if (a <= b) low = std::min(low, (long)(ph.path[(size_t)(PP - 1) * ph.meta.nmap + m] & 0xfffffu) - (b - a + 2));
            }
        }
        const TreeClass &c = th.cls;
        printf("%d %llu %d %d %zu %ld\n", PP, (unsigned long long)q.nmap, c.n_parts, c.items_per_conf, tree_smem_bytes(c), low);
    }
    return 0;
}
