// Which calls take the grouped form of the tree kernel (test_tree_tasks.py; no GPU is needed).  Arguments: layers, window delta, nodes per
// type, node size, policies, configurations of the classes (1, 2, 4, ... stages), then pairs: first configuration, how many.
// Prints parts and group of every class, then per pair 0 or 1 for a pass and for a search.
#include "../paper_2609_39350_b200/csrc/hap_tree_host.h"

#include <cstdio>
#include <cstdlib>

using namespace hap;

int main(int argc, char **argv)
{
    if (argc < 7) return 2;
    const i64 P[4] = {400000, 250000, 200000, 150000};
    DevConst dc{};
    dc.N = atoi(argv[1]); dc.delta_q = atoi(argv[2]); dc.R = 2; dc.tau_linear = 1;
    i64 W = 0;
    for (char *s = strtok(argv[3], ","); s && dc.T < HAP_MAX_TYPES; s = strtok(nullptr, ",")) {
        const int h = dc.T++;
        dc.node_size[h] = atoi(argv[4]); dc.m[h] = (i64)atoi(s) * dc.node_size[h]; dc.P[h] = P[h]; dc.cap_eff[h] = 64ll << 30;
        W += dc.m[h];
    }
    std::vector<TreeClass> cls;
    std::vector<std::shared_ptr<const TreeClassHost>> trees;
    u32 p_lo = 0;
    int PP = 1;
    for (char *s = strtok(argv[6], ","); s; s = strtok(nullptr, ","), PP *= 2) {
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
        in.dc = &dc; in.rep = q; in.n_conf = (size_t)atoi(s); in.n_sm = 148; in.want_tree = true;
        auto th = std::make_shared<TreeClassHost>();
        TreeBuilder(in).build(*th);
        if (!th->ok) return 3;
        th->cls.n_conf = (u32)in.n_conf; th->cls.p_lo = p_lo;
        p_lo += (u32)in.n_conf;
        cls.push_back(th->cls);
        trees.push_back(th);
    }
    tree_policy_items(cls, trees, 148, atoi(argv[5]));
    for (const TreeClass &c : cls) printf("%d %d\n", c.n_parts, c.group);
    for (int a = 7; a + 1 < argc; a += 2)
        for (bool search : {false, true})
            printf("%d\n", (int)tree_grouped(cls, (unsigned)atoi(argv[a]), (unsigned)(atoi(argv[a]) + atoi(argv[a + 1])), 148, search));
    return 0;
}
