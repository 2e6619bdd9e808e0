// Host side of the prefix trees: the mappings of a PP class, their windows and bands, the tree's split into parts and the
// task lists that tree_dp_kernel walks.  Everything here depends on the cluster, the stage count, the layer kinds and
// the window only, never on the profiled tables.
#pragma once
#include "hap_tree.cuh"

#include <algorithm>
#include <cstring>
#include <memory>
#include <unordered_map>
#include <vector>

namespace hap {

struct TreePartHost {
    TreePart meta{};                        // pointers are filled in at the upload
    std::vector<TreeTask> tasks;
    std::vector<u32> path, leaf;
};

struct TreeClassHost {
    bool ok = false;                        // false: the class runs one warp per candidate
    unsigned masks_used = 0xffffffffu;      // type masks that occur (the general kernel builds rows for those only)
    TreeClass cls{};
    double work = 0, chain = 0;             // instructions of a configuration's parts, of its longest part (one policy)
    std::vector<TreePartHost> parts;
};

struct TreeInputs {
    const DevConst *dc;                     // N, T, m, node_size, P, cap_eff, kind_uniform_from, delta_q, uniform, R, tau_linear
    hap_pconf rep;                          // any configuration of the class
    size_t n_conf;
    int n_sm;
    bool want_tree;
};

constexpr u64 kTreeMaxMappings = 1u << 18;
constexpr size_t kSmemPerSm = 227 * 1024;
constexpr size_t kTreeSmemMost = 200 * 1024;     // dynamic part of a block
constexpr size_t kTreeSmemFixed = 64, kTreeSmemStatic = 1024 + 256;     // behind the slices; static variables and the system's part

// shared memory that computing a record takes beside it: layer costs of every type, byte prefixes (mixed kinds)
inline size_t tree_record_scratch(const TreeClass &cl, int N, int T) { return (size_t)T * N * 16 + (cl.all_flat ? 0 : ((size_t)(N + 1) * 17 + 15) / 16 * 16); }

// Cycles a class takes, roughly, in a given number of parts: its instructions at the rate at which the busy warps of an SM issue
// them, then the chain of one item.  Measured on B200: a warp of these kernels issues an instruction every six to seven cycles
// (7.3 warps stand for every issue), an SM 2.3 a cycle when all its warps are busy (57 % of the slots); warps of a block without
// a part still hold their registers.  About two fifths of a class's configurations are feasible (1,024 devices: 27 %, 256
// devices: 41 %).  An item's record comes in between two barriers of its block, 1,500 cycles and one per 16 bytes.  Other
// items fill about half of a chain: counted in full, 32 devices of three types (31 layers) take 79 us instead of 71, a third of it
// 1,024 devices 416 instead of 390, the rest the same.  A pass at 1,024 devices without a homogeneous class, by the parts of
// its 24 mappings at 32 stages (all policies an item): 1 part 527 us, 2 384, 3 351, 4 310, 6 329, 8 324.  Negative: no block fits.
struct TreeWork { double total = 0, longest = 0, n_conf = 0; size_t slice = 0; u32 rec_bytes = 0; int n_parts = 0, n_sm = 0; };
constexpr double kTreeIssue = 2.3, kTreeWarpIssue = 0.15, kTreeLive = 0.4, kTreeChain = 0.5;
// Warp instructions: of an iteration of tasks of 1, 2 or 4 end layers and of a length in it; of 32 last stages and of a stage
// on the way back.
constexpr double kTreeIteration[3] = {70.0, 90.0, 130.0}, kTreePerLength[3] = {15.0, 24.0, 41.0}, kTreeLeaf = 150.0, kTreePerStage = 100.0;
inline double tree_time(const TreeWork &w, double busy_issue)
{
    const double copy = 1500.0 + w.rec_bytes / 16, live = kTreeLive * w.n_conf;
    return live * (w.total + copy * kTreeWarpIssue * w.n_parts) / (w.n_sm * busy_issue) + kTreeChain * (w.longest / kTreeWarpIssue + copy);
}
inline double tree_time(const TreeWork &w)
{
    const size_t smem = w.rec_bytes + kTreeWarps * w.slice + kTreeSmemFixed;
    const int per_sm = (int)std::min<size_t>(kTreeBlocksPerSm, kSmemPerSm / (smem + kTreeSmemStatic)), items = (w.n_parts + kTreeWarps - 1) / kTreeWarps;
    if (per_sm < 1 || smem > kTreeSmemMost) return -1.0;
    return tree_time(w, std::min(kTreeIssue, per_sm * ((double)w.n_parts / items) * kTreeWarpIssue));
}

class TreeBuilder {
public:
    explicit TreeBuilder(const TreeInputs &in) : in_(in), dc_(*in.dc), N_(in.dc->N), PP_(in.rep.PP), T_(in.dc->T) {}

    void build(TreeClassHost &out)
    {
        nmap_ = in_.rep.nmap;
        if (nmap_ == 0 || nmap_ > kTreeMaxMappings) return;
        decode();
        out.masks_used = 0;
        for (size_t q = 0; q < mask_.size(); ++q) out.masks_used |= 1u << mask_[q];
        if (!in_.want_tree || !windows()) return;
        Part all;
        out.ok = class_fields(out.cls, all) && split(out, all);
    }

private:
    struct Node { u32 parent, rowoff; uint8_t mask, link, nmin, nmax; int bl, bh; };
    struct Part {
        u64 m0, m1;
        std::vector<std::vector<Node>> lv;
        std::vector<u32> leaf_node;
        std::vector<u64> order; std::vector<u32> place; std::vector<Node> sorted;      // (kept: a cluster asks for thousands of parts)
    };

    // the class's mappings in enumeration order (decode_stage unranks single ones; here they follow one another)
    void decode()
    {
        mask_.resize((size_t)nmap_ * PP_); link_.resize((size_t)nmap_ * PP_);
        if (in_.rep.mode != HAP_MAP_MULTISET) {
            for (u64 m = 0; m < nmap_; ++m)
                for (int s = 0; s < PP_; ++s) {
                    const StageMap sm = decode_stage(dc_, in_.rep, m, s);
                    mask_[(size_t)m * PP_ + s] = (uint8_t)sm.mask;
                    link_[(size_t)m * PP_ + s] = (uint8_t)(s > 0 ? (sm.cls | (sm.ha << 2) | (sm.hb << 4)) : 0);
                }
            return;
        }
        const i64 G = in_.rep.G;
        std::vector<uint8_t> seq;
        std::vector<uint8_t> same[HAP_MAX_TYPES];               // link class into the q-th stage of a type from the one before it
        for (int h = 0; h < T_; ++h) {
            const int cnt = (int)(dc_.m[h] / G);
            for (int q = 0; q < cnt; ++q) {
                seq.push_back((uint8_t)h);
                const i64 first = (i64)q * G;
                same[h].push_back((first - 1) / dc_.node_size[h] == first / dc_.node_size[h] ? HAP_INTRA : HAP_INTER);
            }
        }
        u64 m = 0;
        do {
            int used[HAP_MAX_TYPES] = {0, 0, 0, 0};
            for (int s = 0; s < PP_; ++s) {
                const int h = seq[s], q = used[h]++;
                mask_[(size_t)m * PP_ + s] = (uint8_t)(1 << h);
                const int cls = s == 0 ? 0 : seq[s - 1] != h ? HAP_CROSS : same[h][q];
                link_[(size_t)m * PP_ + s] = (uint8_t)(s > 0 ? (cls | (seq[s - 1] << 2) | (h << 4)) : 0);
            }
            ++m;
        } while (m < nmap_ && std::next_permutation(seq.begin(), seq.end()));
    }

    // load-balance window of every stage and band of reachable end layers, by the formulas of pipeline_dp_kernel
    bool windows()
    {
        nmin_.resize(mask_.size()); nmax_.resize(mask_.size()); bl_.resize(mask_.size()); bh_.resize(mask_.size()); dead_.assign((size_t)nmap_, 0);
        i64 Pmin[1 << HAP_MAX_TYPES] = {0};
        for (int mk = 1; mk < (1 << T_); ++mk) {
            bool seen = false, capseen = false;
            i64 cap = 0;
            for (int h = 0; h < T_; ++h)
                if (mk >> h & 1) {
                    if (!seen || dc_.P[h] < Pmin[mk]) Pmin[mk] = dc_.P[h];
                    if (!capseen || dc_.cap_eff[h] < cap) { cap = dc_.cap_eff[h]; capt_[mk] = h; }
                    seen = capseen = true;
                }
        }
        // the window of a stage depends on its type mask and on the mapping's summed compute power only
        i64 win_Ps = -1;
        int win_lo[1 << HAP_MAX_TYPES], win_hi[1 << HAP_MAX_TYPES];
        std::vector<int> lo(PP_), hi(PP_);
        for (u64 m = 0; m < nmap_; ++m) {
            const size_t at = (size_t)m * PP_;
            i64 Ps = 0;
            for (int s = 0; s < PP_; ++s) {
                const int mk = mask_[at + s];
                if (mk < 1 || mk >= (1 << T_)) return false;
                Ps += Pmin[mk];
            }
            if (!dc_.uniform && dc_.delta_q >= 0 && Ps != win_Ps) {
                const i64 den = 1024 * Ps;
                for (int mk = 1; mk < (1 << T_); ++mk) {
                    i64 a = ((i64)(1024 - dc_.delta_q) * Pmin[mk] * N_) / den;
                    i64 b = ((i64)(1024 + dc_.delta_q) * Pmin[mk] * N_ + den - 1) / den;
                    if (a < 1) a = 1;
                    if (b > N_ - PP_ + 1) b = N_ - PP_ + 1;
                    win_lo[mk] = (int)a; win_hi[mk] = (int)b;
                }
                win_Ps = Ps;
            }
            int tmin = 0, tmax = 0;
            for (int s = 0; s < PP_; ++s) {
                lo[s] = 1; hi[s] = N_ - PP_ + 1;
                if (dc_.uniform) { lo[s] = N_ / PP_; hi[s] = (N_ + PP_ - 1) / PP_; }
                else if (dc_.delta_q >= 0) { lo[s] = win_lo[mask_[at + s]]; hi[s] = win_hi[mask_[at + s]]; }
                if (lo[s] < 0 || lo[s] > 255 || hi[s] < 0 || hi[s] > 255) return false;
                tmin += lo[s]; tmax += hi[s];
            }
            int smin = 0, smax = 0;
            for (int s = 0; s < PP_; ++s) {
                smin += lo[s]; smax += hi[s];
                int a = std::max(smin, s + 1), b = std::min(smax, N_ - PP_ + s + 1);
                a = std::max(a, N_ - (tmax - smax)); b = std::min(b, N_ - (tmin - smin));
                if (a > b) dead_[m] = 1;
                nmin_[at + s] = (uint8_t)lo[s]; nmax_[at + s] = (uint8_t)hi[s];
                bl_[at + s] = (uint8_t)std::max(0, std::min(255, a)); bh_[at + s] = (uint8_t)std::max(0, std::min(255, b));
            }
        }
        shared_.assign((size_t)nmap_, 0);
        for (u64 m = 0, before = nmap_; m < nmap_; ++m) {
            if (dead_[m]) continue;
            if (before < nmap_) {
                const size_t a = (size_t)before * PP_, b = (size_t)m * PP_;
                int d = 0;
                while (d < PP_ && mask_[a + d] == mask_[b + d] && link_[a + d] == link_[b + d] && nmin_[a + d] == nmin_[b + d] && nmax_[a + d] == nmax_[b + d]) ++d;
                shared_[m] = (uint8_t)d;
            }
            before = m;
        }
        return true;
    }

    // distinct stage prefixes of mappings [m0, m1); a node's band is the union over the mappings below it, which only adds
    // cells that hold their plain recurrence value
    void nodes(u64 m0, u64 m1, Part &pt) const
    {
        pt.m0 = m0; pt.m1 = m1;
        pt.lv.resize(PP_ + 1);
        for (auto &v : pt.lv) v.clear();
        pt.leaf_node.assign((size_t)(m1 - m0), 0);
        u32 path[HAP_MAX_PP + 1] = {0};
        uint8_t lo[HAP_MAX_PP], hi[HAP_MAX_PP];                 // bands of the path's nodes, by stage
        int open = 0;                                           // stages of the path that have a node
        auto close = [&](int from) { for (int s = from; s < open; ++s) { Node &nd = pt.lv[s + 1][path[s + 1]]; nd.bl = lo[s]; nd.bh = hi[s]; } };
        for (u64 m = m0; m < m1; ++m) {
            if (dead_[m]) continue;
            const size_t at = (size_t)m * PP_;
            const int same = std::min(open, (int)shared_[m]);
            close(same);
            for (int s = 0; s < same; ++s) { lo[s] = std::min(lo[s], bl_[at + s]); hi[s] = std::max(hi[s], bh_[at + s]); }
            for (int s = same; s < PP_ - 1; ++s) {
                lo[s] = bl_[at + s]; hi[s] = bh_[at + s];
                path[s + 1] = (u32)pt.lv[s + 1].size();
                pt.lv[s + 1].push_back(Node{s ? path[s] : 0, 0, mask_[at + s], link_[at + s], nmin_[at + s], nmax_[at + s], 0, 0});
            }
            open = PP_ - 1;
            pt.leaf_node[(size_t)(m - m0)] = PP_ > 1 ? path[PP_ - 1] : 0;
        }
        close(0);
        // nodes of a depth by the width of their band, then of their window (widest first): the lanes of a warp get runs of
        // similar length
        for (int d = 1; d < PP_; ++d) {
            std::vector<Node> &lv = pt.lv[d];
            const size_t n = lv.size();
            auto key = [&](size_t i) { return (u32)(512 - (lv[i].bh - lv[i].bl)) << 16 | (u32)(512 - ((int)lv[i].nmax - (int)lv[i].nmin)); };
            u32 c = kTreeAhead;
            auto put = [&](Node &nd) { c += kTreePad; nd.rowoff = c; c += (u32)(nd.bh - nd.bl + 1); };
            size_t sorted = 1;
            while (sorted < n && key(sorted - 1) <= key(sorted)) ++sorted;
            if (sorted >= n) {                                  // (as they come)
                for (Node &nd : lv) put(nd);
                continue;
            }
            pt.order.resize(n); pt.place.resize(n); pt.sorted.resize(n);
            for (size_t i = 0; i < n; ++i) pt.order[i] = (u64)key(i) << 32 | i;
            std::sort(pt.order.begin(), pt.order.end());
            for (size_t i = 0; i < n; ++i) {
                const u32 from = (u32)pt.order[i];
                put(pt.sorted[i] = lv[from]);
                pt.place[from] = (u32)i;
            }
            lv.swap(pt.sorted);
            if (d + 1 < PP_) for (auto &ch : pt.lv[d + 1]) ch.parent = pt.place[ch.parent];
            else for (u64 m = m0; m < m1; ++m) if (!dead_[m]) pt.leaf_node[(size_t)(m - m0)] = pt.place[pt.leaf_node[(size_t)(m - m0)]];
        }
    }

    int kidx(int d, uint8_t mask, uint8_t link, const TreeClass &cl) const
    {
        const int cls = link & 3, ha = (link >> 2) & 3, hb = (link >> 4) & 3;
        return d == 1 ? cl.mrow_of[mask] : 16 + hb * 6 + (cls == HAP_CROSS ? 2 + ha : cls);
    }

    // row groups, windows, thresholds and the layout of a configuration's record
    bool class_fields(TreeClass &cl, Part &all)
    {
        const int R = dc_.R;
        cl.PP = PP_;
        std::memset(cl.mrow_of, 255, sizeof(cl.mrow_of));
        unsigned used = 0;
        for (size_t q = 0; q < mask_.size(); ++q) used |= 1u << mask_[q];
        for (int mk = 1; mk < (1 << T_); ++mk)
            if ((used >> mk) & 1u) { cl.mrow_of[mk] = (uint8_t)cl.n_mrows; cl.mask_of_row[cl.n_mrows] = (uint8_t)mk; cl.n_mrows++; }
        nodes(0, nmap_, all);
        std::memset(cl.first_min, 255, sizeof(cl.first_min));
        for (int d = 1; d <= PP_; ++d) { cl.jlo[d] = 255; cl.jhi[d] = 0; cl.kmin[d] = 255; cl.kmax[d] = 0; }
        auto see_split = [&](int d, int j, const Node &nd, int pbl, int pbh) {
            const int klo = std::max(j - (int)nd.nmax, pbl), khi = std::min(j - (int)nd.nmin, pbh);
            if (klo > khi) return;
            cl.kmin[d] = (uint8_t)std::min<int>(cl.kmin[d], klo); cl.kmax[d] = (uint8_t)std::max<int>(cl.kmax[d], khi);
        };
        for (int d = 1; d < PP_; ++d)
            for (const Node &nd : all.lv[d]) {
                const int t = capt_[nd.mask];
                cl.jlo[d] = (uint8_t)std::min<int>(cl.jlo[d], nd.bl); cl.jhi[d] = (uint8_t)std::max<int>(cl.jhi[d], nd.bh);
                cl.wmax[d] = std::max(cl.wmax[d], nd.nmax);
                cl.tmask[d] |= (uint8_t)(1u << t);
                if (d == 1) cl.first_min[t] = (uint8_t)std::min<int>(cl.first_min[t], nd.bl);
                const int pbl = d > 1 ? all.lv[d - 1][nd.parent].bl : 0, pbh = d > 1 ? all.lv[d - 1][nd.parent].bh : 0;
                for (int j = nd.bl; j <= nd.bh; ++j) see_split(d, j, nd, pbl, pbh);
            }
        cl.jlo[PP_] = cl.jhi[PP_] = (uint8_t)N_;
        for (u64 m = 0; m < nmap_; ++m) {
            if (dead_[m]) continue;
            const size_t at = (size_t)m * PP_ + PP_ - 1;
            const int t = capt_[mask_[at]];
            cl.wmax[PP_] = std::max(cl.wmax[PP_], nmax_[at]);
            cl.tmask[PP_] |= (uint8_t)(1u << t);
            if (PP_ == 1) cl.first_min[t] = (uint8_t)N_;
            Node lf{};
            lf.nmin = nmin_[at]; lf.nmax = nmax_[at];
            const int pbl = PP_ > 1 ? all.lv[PP_ - 1][all.leaf_node[(size_t)m]].bl : 0, pbh = PP_ > 1 ? all.lv[PP_ - 1][all.leaf_node[(size_t)m]].bh : 0;
            see_split(PP_, N_, lf, pbl, pbh);
        }
        // A depth whose cells only look at splits behind the last change of layer kind sees spans of one kind only: their
        // memory depends on the length alone.  All depths of a model whose layers are all of one kind; every depth but the
        // first few of a model with a dense prefix.
        u32 nf = 0;
        cl.all_flat = 1;
        for (int d = 1; d <= PP_; ++d) {
            cl.flat[d] = (cl.kmin[d] > cl.kmax[d] || (int)cl.kmin[d] >= dc_.kind_uniform_from) ? 1 : 0;
            if (cl.flat[d]) continue;
            cl.all_flat = 0;
            cl.nf_off[d] = nf; cl.nf_w[d] = (u32)(cl.jhi[d] - cl.jlo[d] + 1);
            nf += (u32)(T_ * R) * cl.nf_w[d];
        }
        auto up16 = [](u32 v) { return (v + 15) / 16 * 16; };
        const int RW = dc_.tau_linear ? R : 2;
        cl.o_rows = kTreeOffMinfo + (u32)(cl.n_mrows * kTreeMinfo * 8);
        cl.o_thr_nf = up16(cl.o_rows + (u32)(cl.n_mrows * RW * (N_ + 1) * 8));
        cl.rec_bytes = up16(cl.o_thr_nf + nf);
        return true;
    }

    // a task before it is laid out: end layers j .. j + cnt - 1 of a node, stage lengths a .. b (b = a - 1: none)
    struct Piece {
        u32 node;
        uint8_t j, cnt, a, b;
        int length() const { return (int)b + 1 - (int)a; }
    };

    // What one depth after the other is cut with.
    struct Cutter {
        std::vector<Piece> tasks, rest, scratch;
        std::vector<int16_t> len[3];                            // lengths of tasks of 1, 2 and 4 end layers, room for eight behind the last
        size_t n[3];
        u32 of[257] = {0};                                      // how many are of a length: all zero between uses
        std::unordered_map<u64, double> known;                  // times by a hash of the depth's nodes (of which parts have many in common)

        // Warp instructions of the first `most` of the tasks of J end layers, the longest ones first, 32 an iteration.
        double time(int J, size_t most)
        {
            const int16_t *v = len[J / 2].data(), *end = v + n[J / 2];
            const double it = kTreeIteration[J / 2], per = kTreePerLength[J / 2];
            int16_t hi = 0;
            for (const int16_t *l = v; l < end; ++l) hi = std::max(hi, *l);
            if (n[J / 2] <= 32) return most ? it + per * std::max<int>(1, hi) : 0.0;
            for (const int16_t *l = v; l < end; ++l) ++of[*l];
            double t = 0;
            size_t at = 0, next = 0;                            // tasks of length l or more; the first of the next iteration
            for (int l = hi; l >= 0; --l) {
                for (at += of[l]; next < at && next < most; next += 32) t += it + per * std::max(1, l);
                of[l] = 0;
            }
            return t;
        }

        // longest first, equal ones in the order they had
        void sort(std::vector<Piece> &v, size_t from)
        {
            int hi = 0;
            for (size_t q = from; q < v.size(); ++q) { const int l = v[q].length(); ++of[l]; hi = std::max(hi, l); }
            u32 at = 0;
            for (int l = hi; l >= 0; --l) { const u32 k = of[l]; of[l] = at; at += k; }
            scratch.resize(v.size() - from);
            for (size_t q = from; q < v.size(); ++q) scratch[of[v[q].length()]++] = v[q];
            std::copy(scratch.begin(), scratch.end(), v.begin() + (std::ptrdiff_t)from);
            std::memset(of, 0, ((size_t)hi + 1) * sizeof(u32));
        }
    };

    // a node with the end layers of the one before it
    struct Reach {
        int nmin, nmax, pbl, pbh;
        // shortest and longest stage that end at j .. j + J - 1 and reach the row before
        int a(int j) const { return std::max(nmin, j - pbh); }
        int b(int j, int J) const { return std::min(nmax, j + J - 1 - pbl); }
        int length(int j, int J) const { return std::max(0, b(j, J) - a(j) + 1); }
        Piece piece(u32 node, int j, int J) const { return Piece{node, (uint8_t)j, (uint8_t)J, (uint8_t)a(j), (uint8_t)(a(j) + length(j, J) - 1)}; }
    };
    static Reach reach(const Part &pt, int d, u32 ni)
    {
        const Node &nd = pt.lv[d][ni];
        if (d == 1) return Reach{nd.nmin, nd.nmax, 0, 0};
        const Node &pn = pt.lv[d - 1][nd.parent];
        return Reach{nd.nmin, nd.nmax, pn.bl, pn.bh};
    }

    // lengths of the tasks of J end layers of a depth, node by node (eight at a time: what lies behind a node's last one is written over)
    template <int J>
    static void lengths(const Part &pt, int d, Cutter &c)
    {
        size_t n = 0;
        for (const Node &nd : pt.lv[d]) n += (size_t)std::max(0, nd.bh - nd.bl + J) / J;
        c.n[J / 2] = n;
        if (c.len[J / 2].size() < n + 8) c.len[J / 2].resize(2 * n + 8);
        int16_t *o = c.len[J / 2].data();
        for (u32 ni = 0; ni < pt.lv[d].size(); ++ni) {
            const Reach r = reach(pt, d, ni);
            const int16_t bh = (int16_t)pt.lv[d][ni].bh, nmin = (int16_t)(r.nmin - 1), nmax = (int16_t)r.nmax, pbl = (int16_t)r.pbl, pbh = (int16_t)(r.pbh + 1);
            for (int j = pt.lv[d][ni].bl; j <= bh; j += 8 * J) {
                for (int k = 0; k < 8; ++k) {
                    const int16_t first = (int16_t)(j + k * J), last = std::min<int16_t>((int16_t)(first + J - 1), bh);
                    const int16_t b = std::min<int16_t>(nmax, (int16_t)(last - pbl)), a = std::max<int16_t>(nmin, (int16_t)(first - pbh));
                    o[k] = std::max<int16_t>(0, (int16_t)(b - a));
                }
                o += std::min(8, (bh - j + J) / J);
            }
        }
    }

    // lengths of the last `left` tasks of four end layers, in the order of their lengths, as tasks of one and two: the shortest ones, the
    // last of the list where they are alike
    static void rest_lengths(const Part &pt, int d, Cutter &c, size_t left)
    {
        const int16_t *len = c.len[2].data() + c.n[2];
        int most = 0, hi = 0;
        for (size_t q = 0; q < c.n[2]; ++q) { const int l = c.len[2][q]; ++c.of[l]; hi = std::max(hi, l); }
        size_t equal = left;                                    // of length `most`
        for (; c.of[most] < equal; ++most) equal -= c.of[most];
        std::memset(c.of, 0, ((size_t)hi + 1) * sizeof(u32));
        for (int J : {1, 2}) if (c.len[J / 2].size() < (size_t)kTreeJ / J * left + 8) c.len[J / 2].resize((size_t)kTreeJ / J * left + 8);
        int16_t *one = c.len[0].data(), *two = c.len[1].data();
        for (u32 ni = (u32)pt.lv[d].size(); left && ni-- > 0;) {
            const Reach r = reach(pt, d, ni);
            const int bl = pt.lv[d][ni].bl, bh = pt.lv[d][ni].bh;
            for (int j = bl + (bh - bl) / kTreeJ * kTreeJ; left && j >= bl; j -= kTreeJ) {
                const int l = *--len;
                if (l > most || (l == most && equal == 0)) continue;
                if (l == most) --equal;
                --left;
                const int end = std::min(bh, j + kTreeJ - 1);
                for (int i = j; i <= end; i += 2) {
                    *two++ = (int16_t)r.length(i, std::min(2, end - i + 1));
                    *one++ = (int16_t)r.length(i, 1);
                    if (i < end) *one++ = (int16_t)r.length(i + 1, 1);
                }
            }
        }
        c.n[0] = (size_t)(one - c.len[0].data()); c.n[1] = (size_t)(two - c.len[1].data());
    }

    // The tasks of a depth, 32 an iteration, and the warp instructions they take.  Four end layers a task are cheapest where the lanes are
    // full: a length's loads, tests and steps serve four splits.  What does not fill an iteration, often the whole depth, is cut
    // into tasks of two or one, which take a fraction of the instructions on lanes that would idle.  Longest tasks first, so
    // that an iteration's are alike.  Depths whose thresholds go by end layer take one each.  Against tasks of four everywhere (20
    // of 32 lanes active, now 25): a pass at 1,024 devices 390 -> 378 us, 256 devices with partitions 473 -> 439, 64 devices with three
    // levels 150 -> 130, search at 1,024 devices 233 -> 220.
    // `lay`: leaves the tasks in the order a warp takes them.  The search for the number of parts asks for the time alone, thousands of
    // times a cluster: it follows from how many tasks are of a length, and nothing is put in order.
    double cut(const Part &pt, int d, bool flat, Cutter &c, bool lay) const
    {
        u64 hash = flat ? 1469598103934665603ull : 1099511628211ull;
        if (!lay) {
            for (u32 ni = 0; ni < pt.lv[d].size(); ++ni) {
                const Reach r = reach(pt, d, ni);
                const Node &nd = pt.lv[d][ni];
                hash = (hash ^ ((u64)r.nmin << 40 | (u64)r.nmax << 32 | (u64)r.pbl << 24 | (u64)r.pbh << 16 | (u64)nd.bl << 8 | (u64)nd.bh)) * 0x9e3779b97f4a7c15ull;
                hash ^= hash >> 29;
            }
            const auto it = c.known.find(hash);
            if (it != c.known.end()) return it->second;
        }
        const int J0 = flat ? kTreeJ : 1;
        if (flat) lengths<kTreeJ>(pt, d, c);
        else lengths<1>(pt, d, c);
        const size_t n = c.n[J0 / 2], full = n / 32 * 32;
        double best = c.time(J0, n);
        size_t head = n;
        int width = kTreeJ;
        if (flat)
            for (size_t h : {full, (size_t)0}) {                // tasks of four end layers that stay: whole iterations, or none
                if (h < n && (n - h) * 2 <= 96) {               // (two full iterations more than one: no gain)
                    if (h) rest_lengths(pt, d, c, n - h);
                    else {
                        if (n * 4 <= 96) lengths<1>(pt, d, c);
                        lengths<2>(pt, d, c);
                    }
                    const double before = h ? c.time(kTreeJ, h) : 0.0;
                    for (int J : {2, 1}) {
                        if ((n - h) * (size_t)(kTreeJ / J) > 96) continue;
                        const double t = before + c.time(J, c.n[J / 2]);
                        if (t < best) { best = t; head = h; width = J; }
                    }
                }
                if (full == 0) break;
            }
        if (!lay) { c.known.emplace(hash, best); return best; }
        std::vector<Piece> &out = c.tasks;
        out.clear();
        for (u32 ni = 0; ni < pt.lv[d].size(); ++ni) {
            const Reach r = reach(pt, d, ni);
            const int bh = pt.lv[d][ni].bh;
            for (int j = pt.lv[d][ni].bl; j <= bh; j += J0) out.push_back(r.piece(ni, j, std::min(J0, bh - j + 1)));
        }
        c.sort(out, 0);
        if (head < n) {
            c.rest.assign(out.begin() + (std::ptrdiff_t)head, out.end());
            out.resize(head);
            for (const Piece &t : c.rest) {
                const Reach r = reach(pt, d, t.node);
                for (int i = 0; i < t.cnt; i += width) out.push_back(r.piece(t.node, t.j + i, std::min(width, t.cnt - i)));
            }
            c.sort(out, head);
        }
        return best;
    }

    // warp instructions of a part, roughly: what the split is chosen by
    double cost(const Part &pt, const TreeClass &cl, Cutter &cutter) const
    {
        double total = (double)((pt.m1 - pt.m0 + 31) / 32) * (kTreeLeaf + kTreePerStage * PP_);
        for (int d = 1; d < PP_; ++d) total += cut(pt, d, cl.flat[d] != 0, cutter, false);
        return total;
    }

    // a warp's row buffers and choices for it, in bytes
    size_t slice(const Part &pt) const
    {
        u32 cells[2] = {0, 0}, ch = 0;
        for (int d = 1; d < PP_; ++d) {
            u32 c = kTreeAhead + kTreePad;
            for (const Node &nd : pt.lv[d]) c += (u32)(nd.bh - nd.bl + 1) + kTreePad;
            cells[d & 1] = std::max(cells[d & 1], c); ch += c;
        }
        return ((size_t)((cells[0] + 1) / 2 * 2) + (cells[1] + 1) / 2 * 2) * 8 + (ch + 15) / 16 * 16;
    }

    bool split(TreeClassHost &out, const Part &all)
    {
        // Parts over contiguous ranges of mappings: the few nodes near the root that two parts share are computed by both, so
        // smaller parts cost little; more parts shorten the longest chain and fill the warps of a block, fewer fill the lanes
        // of a warp better.  How many is what tree_time says: a guess, then every number from the first one that may be better.  (Climbing from
        // the guess alone took a fifth less time and ended at other, slower numbers: how many blocks an SM holds grows in steps.)
        TreeClass &cl = out.cls;
        Cutter cutter;
        Part pt;
        constexpr int counts[] = {1, 2, 3, 4, 6, 8, 12, 16, 20, 24, 28, 32, 40, 48, 56, 64, 80, 96, 128, 192, 256, 384, 512, 768, 1024, 2048, 4096, 8192};
        constexpr int n_counts = (int)(sizeof(counts) / sizeof(counts[0]));
        int last = 0;
        while (last + 1 < n_counts && (u64)counts[last + 1] <= nmap_) ++last;
        // What the whole tree takes says where to look first, and which numbers are too small: parts take their share of it at least (but
        // for how full their iterations are and how narrow their bands), and an iteration a depth, an end and a way back.
        const double least = (PP_ - 1) * (kTreeIteration[0] + kTreePerLength[0]) + kTreeLeaf + kTreePerStage * PP_;
        TreeWork w;
        w.n_conf = (double)in_.n_conf; w.n_sm = in_.n_sm; w.rec_bytes = cl.rec_bytes;
        const double whole = cost(all, cl, cutter);
        const size_t whole_slice = slice(all);
        double bound[n_counts], guess = -1.0;
        int at = last;
        for (int i = 0; i <= last; ++i) {
            w.n_parts = counts[i]; w.slice = whole_slice / (size_t)counts[i];
            w.longest = whole / counts[i] + least; w.total = w.longest * counts[i];
            const double t = tree_time(w);
            if (t > 0 && (guess < 0 || t < guess)) { guess = t; at = i; }
            w.slice = w.slice / 4 * 3;
            w.longest = std::max(0.85 * whole / counts[i], least); w.total = 0.85 * whole;
            bound[i] = tree_time(w);
        }
        double best = -1.0;
        int best_at = -1;
        cl.n_parts = 0;
        // takes counts[i] parts if that is faster than what is taken; true: more parts are not
        auto look = [&](int i) {
            const u64 np = (u64)counts[i];
            w.n_parts = (int)np; w.slice = 0; w.total = w.longest = 0.0;
            double t = tree_time(w);
            u64 q = 0;
            while (q < np && t > 0 && (best < 0 || t <= best)) {
                nodes(nmap_ * q / np, nmap_ * (q + 1) / np, pt);
                w.slice = std::max(w.slice, slice(pt));
                const double c = cost(pt, cl, cutter);
                w.total += c; w.longest = std::max(w.longest, c);
                t = tree_time(w);
                ++q;
            }
            if (t <= 0) return false;                           // (no block has room for a part of that size)
            if (best < 0 || (q == np && (t < best || (t == best && i < best_at)))) { best = t; best_at = i; cl.n_parts = (int)np; out.work = w.total; out.chain = w.longest; }
            // finer parts share no more prefixes: what they all cost only grows, but for how full their iterations are.  A sum of a growing and
            // a falling term has one minimum, but for the rounding to whole warps: half as much again lies behind it
            TreeWork finer = w;
            finer.total *= (double)np / (double)q;
            t = std::max(t, tree_time(finer));
            finer.total *= 0.85; finer.longest = least;
            return tree_time(finer, kTreeIssue) > best || (t > 1.5 * best && best_at != i);
        };
        look(at);
        for (int i = 0; i <= last; ++i)
            if (i != at && bound[i] > 0 && (best < 0 || bound[i] < best) && look(i) && i > best_at) break;
        if (!cl.n_parts) return false;                          // no part leaves room for a block
        cl.items_per_conf = (cl.n_parts + kTreeWarps - 1) / kTreeWarps;
        cl.ipc_inverse = cl.items_per_conf > 1 ? (u32)(((1ull << 32) + cl.items_per_conf - 1) / (u64)cl.items_per_conf) : 0u;
        cl.policy_items = 1;
        cl.group = 1;
        out.parts.resize((size_t)cl.n_parts);
        for (int q = 0; q < cl.n_parts; ++q) {
            nodes(nmap_ * q / cl.n_parts, nmap_ * (q + 1) / cl.n_parts, pt);
            if (!emit(pt, cl, cutter, out.parts[(size_t)q])) return false;
        }
        return true;
    }

    // nothing to do beside t (what the 32 tasks of an iteration share, and addresses that exist)
    static TreeTask no_task(const TreeTask &t) { return make_uint4(t.x, (t.y & 255u) | 1u << 8, t.z, t.w); }

    bool emit(const Part &pt, TreeClass &cl, Cutter &cutter, TreePartHost &ph) const
    {
        TreePart &tp = ph.meta;
        const u32 nmap = (u32)(pt.m1 - pt.m0);
        tp.nmap = nmap; tp.m_lo = (u32)pt.m0;
        u32 cells = 0, buf[2] = {0, 0}, cell_lo[HAP_MAX_PP + 1] = {0};      // choices of depth d start at cell_lo[d]
        const std::vector<Piece> &pieces = cutter.tasks;
        for (int d = 1; d < PP_; ++d) {
            cell_lo[d] = cells;
            const size_t first = ph.tasks.size();
            u32 c = kTreeAhead + kTreePad;
            for (const Node &nd : pt.lv[d]) c += (u32)(nd.bh - nd.bl + 1) + kTreePad;
            cut(pt, d, cl.flat[d] != 0, cutter, true);
            int J = 1;
            for (size_t at = 0; at < pieces.size(); ++at) {
                const Piece &q = pieces[at];
                const Node &nd = pt.lv[d][q.node];
                const Node *pn = d > 1 ? &pt.lv[d - 1][nd.parent] : nullptr;
                // slot of the parent's entry 0 (before the first stage: one row of layer 0 behind its padding)
                const int pbl = pn ? pn->bl : 0, porg = pn ? (int)pn->rowoff - pn->bl : kTreeAhead + kTreePad;
                // (no length reaches the parent's row: the origin below only has to be a slot of it)
                const int src = q.a > q.b ? porg + pbl : porg + q.j - q.a, dst = (int)nd.rowoff + q.j - nd.bl;
                if (src < 0 || src > 65535 || dst > 65535 || cells + (u32)dst > 65535) return false;
                TreeTask t;
                t.x = (u32)src | ((u32)dst << 16);
                t.y = (u32)q.j | ((u32)q.a << 8) | ((u32)q.b << 16) | ((u32)q.cnt << 24) | (q.j == nd.bl ? 1u << 27 : 0u) |
                      (q.node + 1 == pt.lv[d].size() && q.j + q.cnt > nd.bh ? 1u << 28 : 0u);
                t.z = (u32)kidx(d, nd.mask, nd.link, cl) | ((u32)cl.mrow_of[nd.mask] << 8) | ((u32)((d - 1) * HAP_MAX_TYPES + capt_[nd.mask]) << 16);
                // tasks of an iteration are of the same number of end layers: that of its largest one
                const size_t it = at / 32 * 32;
                if (at == it) {
                    J = 1;
                    for (size_t x = it; x < std::min(it + 32, pieces.size()); ++x) J = std::max(J, (int)pieces[x].cnt);
                }
                t.w = (cells + (u32)dst) | (u32)(J > 2 ? 4 : J) << 16 | (it + 32 >= pieces.size() ? kTaskEnds : 0u) | (cl.flat[d] ? 0u : kTaskByLayer);
                ph.tasks.push_back(t);
            }
            while ((ph.tasks.size() - first) % 32) ph.tasks.push_back(no_task(ph.tasks.back()));
            buf[d & 1] = std::max(buf[d & 1], c);
            cells += c;
        }
        tp.n_iter = (u32)(ph.tasks.size() / 32);
        const TreeTask behind = no_task(ph.tasks.empty() ? make_uint4(0, 0, 0, 1u << 16) : ph.tasks.back());
        ph.tasks.insert(ph.tasks.end(), 32, behind);
        for (int q = 0; q < 2; ++q) cl.buf_cells[q] = std::max(cl.buf_cells[q], (buf[q] + 1) / 2 * 2);
        cl.ch_bytes = std::max(cl.ch_bytes, (cells + 15) / 16 * 16);
        ph.path.assign((size_t)nmap * PP_, 0);
        ph.leaf.assign(nmap, 1u);                               // a = 1 > b = 0
        for (u32 m = 0; m < nmap; ++m) {
            if (dead_[pt.m0 + m]) continue;
            const size_t at = (size_t)(pt.m0 + m) * PP_;
            u32 nd = PP_ > 1 ? pt.leaf_node[m] : 0;
            // lengths of the last stage that reach the parent's row
            const int pbl = PP_ > 1 ? pt.lv[PP_ - 1][nd].bl : 0, pbh = PP_ > 1 ? pt.lv[PP_ - 1][nd].bh : 0;
            const int a = std::max((int)nmin_[at + PP_ - 1], N_ - pbh), b = std::min((int)nmax_[at + PP_ - 1], N_ - pbl);
            if (a > b) continue;
            ph.leaf[m] = (u32)a | ((u32)b << 8);
            for (int d = PP_; d >= 1; --d) {
                int org = PP_ > 1 ? 0 : kTreeAhead + kTreePad;
                if (d == PP_) { if (PP_ > 1) { const Node &p = pt.lv[PP_ - 1][nd]; org = (int)p.rowoff - p.bl + N_ - a; } }
                else { const Node &p = pt.lv[d][nd]; org = (int)cell_lo[d] + (int)p.rowoff - p.bl + 256; nd = p.parent; }
                ph.path[(size_t)(d - 1) * nmap + m] = (u32)org | ((u32)kidx(d, mask_[at + d - 1], link_[at + d - 1], cl) << 20) |
                                                      ((u32)cl.mrow_of[mask_[at + d - 1]] << 26) | ((u32)capt_[mask_[at + d - 1]] << 30);
            }
        }
        return true;
    }

    const TreeInputs &in_;
    const DevConst &dc_;
    const int N_, PP_, T_;
    u64 nmap_ = 0;
    std::vector<uint8_t> mask_, link_, nmin_, nmax_, bl_, bh_, dead_;
    std::vector<uint8_t> shared_;           // stages that a mapping has in common with the one before it
    int capt_[1 << HAP_MAX_TYPES] = {0};
};

inline size_t tree_smem_bytes(const TreeClass &cl, bool grouped = false)
{
    return (size_t)(grouped ? cl.group : 1) * cl.rec_bytes + kTreeWarps * ((size_t)(cl.buf_cells[0] + cl.buf_cells[1]) * 8 + cl.ch_bytes) + kTreeSmemFixed;
}

inline size_t tree_prep_smem_bytes(const TreeClass &cl, int N, int T)
{
    return cl.rec_bytes + tree_record_scratch(cl, N, T);
}

// Classes whose items take one policy each in a pass: those whose chain, walked policy after policy, is a good part of the pass.
// Measured at 1,024 devices with two policies, six classes of 24 mappings / four of them and one of 840 mappings: no such items
// 290 / 433 us, where a chain is more than a half of what the pass takes at the rate the chip issues 269 / 433, a quarter
// 253 / 423, a tenth 249 / 416, a fiftieth the same.
inline void tree_policy_items(std::vector<TreeClass> &cls, const std::vector<std::shared_ptr<const TreeClassHost>> &trees, int n_sm, int n_rc)
{
    double all = 0;
    for (const auto &th : trees) all += th->work * kTreeLive * th->cls.n_conf / (n_sm * kTreeIssue);
    for (size_t c = 0; c < cls.size(); ++c)
        cls[c].policy_items = trees[c]->chain / kTreeWarpIssue > 0.1 * all ? n_rc : 1;
    // how many configurations of one or two parts can share a block, a warp per part
    for (TreeClass &cl : cls) {
        cl.group = std::max(1, kTreeWarps / cl.n_parts);
        if (tree_smem_bytes(cl, true) + kTreeSmemStatic > kSmemPerSm / kTreeBlocksPerSm) cl.group = 1;
    }
}

// Whether a call over configurations [p_lo, p_hi) takes the grouped form: where a quarter of a pass's items or more, or half of a search's, are
// of classes that share blocks, and there is more than half a wave of items (all configurations counted, feasible or not).  50 passes of 8 to 1,024 devices and their
// halves to sixteenths, grouped against not: up to half a wave 0.95 to 1.06 times as fast, which is the noise, from there to a wave 3 to
// 5 % faster, with more items 5 to 54 %; below a quarter of such items the same within 1 %.  64 devices, three levels and policies, a pass
// 102 us against 121; 256 devices of two types, 400 configurations of 32 stages 56 against 80.
// Searches of several waves lose four blocks an SM (kTreeSearchBlocksPerSm) by it: 149 unpruned ones of half a wave or more, 0.90 to 1.23 times as
// fast where a quarter to a half of the items are such (24 of them), 0.89 to 1.36, on average 1.06, where more are.
inline bool tree_grouped(const std::vector<TreeClass> &cls, unsigned p_lo, unsigned p_hi, int n_sm, bool search)
{
    double items = 0, few = 0;
    for (const TreeClass &cl : cls) {
        const unsigned a = std::max(p_lo, cl.p_lo), b = std::min(p_hi, cl.p_lo + cl.n_conf);
        if (a >= b) continue;
        const double k = (double)(b - a) * cl.items_per_conf * cl.policy_items;
        items += k; few += cl.group > 1 ? k : 0.0;
    }
    return items > 0.5 * n_sm * kTreeBlocksPerSm && (search ? 2.0 : 4.0) * few >= items;
}

}  // namespace hap
