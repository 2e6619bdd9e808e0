"""The tree kernel at the edges of its tasks and parts, against the oracle."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gen import problems  # noqa: E402
from oracle import Oracle, INF  # noqa: E402

NTHREADS = max(1, len(os.sched_getaffinity(0)))

# nodes per type, layers (rows end 0..3 layers into a task of four), levels (repeated fraction), policies, layer kinds
CASES = [
    ((1, 1), 4, (0, 1024), (3,), "uniform"),
    ((2, 2), 9, (0, 1024), (1, 3), "dense_first"),
    ((2, 1, 1), 18, (0, 307, 1024), (1, 3, 7), "dense_first"),         # levels that are not combined into rows
    ((2, 1, 1), 23, (0, 1024, 2048), (7, 5, 4), "mixed"),
    ((1, 1, 1, 1), 16, (0, 1024, 2048, 3072), (15, 9, 6, 1), "uniform"),
    ((3, 1), 25, (0, 200, 700, 1000), (15, 3), "dense_first"),
]


@pytest.mark.parametrize("nodes,N,tau,policies,kinds", CASES)
def test_tree_tasks_and_levels(nodes, N, tau, policies, kinds):
    import paper_2609_39350_b200 as hap
    pb = problems.random_small(40 + N, N=N, T=len(nodes), nodes_per_type=nodes, node_size=2, window=N % 2 == 1, first_dense=kinds == "dense_first")
    if kinds == "mixed":
        pb.kind[3] = 0
    R = len(tau)
    pb.tau_q = np.array(tau, np.int32)
    pb.xi_q = np.array([1024, 512, 200, 64][:R - 1] + [64], np.int32)
    pb.rc_masks = np.array(policies, np.uint32)
    o = Oracle(pb)
    n, best, index, costs, _ = o.search_pconfs(0, 1, threads=NTHREADS, want_costs=True)
    hp = hap.hap_problem_create(pb)
    hap.hap_enumerate(hp)
    out = hap.hap_pipeline_dp(hp, 0, hp.n_cand, partition=True)
    torch.cuda.synchronize()
    got = out["cost"].cpu().numpy()
    bad = np.nonzero(got != costs)[0]
    assert n == hp.n_cand and bad.size == 0, bad[:8]
    part, rec = out["partition"].cpu().numpy(), out["recompute"].cpu().numpy()
    for idx in np.random.default_rng(N).integers(0, o.n_cand, 60).tolist():
        plan, _, _ = o.eval_index(idx)
        if plan["T_iter"] < INF:
            assert part[idx, :plan["PP"]].tolist() == plan["n"] and rec[idx, :plan["PP"]].tolist() == plan["r"], idx
    hap.hap_problem_destroy(hp)
    for prune in (0, 1):                       # in the order of the lists, in the order of the bounds
        hp = hap.hap_problem_create(pb, prune=prune)
        hap.hap_enumerate(hp)
        if best < INF:
            plan, st = hap.hap_search_best(hp)
            assert (plan["index"], plan["T_iter"]) == (index, best)
            assert st["n_evaluated"] + st["n_pruned"] == hp.n_cand
        else:
            with pytest.raises(hap.HapError):
                hap.hap_search_best(hp)
        hap.hap_problem_destroy(hp)


@pytest.mark.parametrize("objective", ["refine", "exact"])
@pytest.mark.parametrize("nodes,N,tau,policies,kinds", CASES)
def test_refined_search_over_listed_candidates(nodes, N, tau, policies, kinds, objective):
    """The search that refines only listed candidates finds what refining every candidate finds."""
    import paper_2609_39350_b200 as hap
    pb = problems.random_small(90 + N, N=N, T=len(nodes), nodes_per_type=nodes, node_size=2, window=N % 2 == 0, first_dense=kinds == "dense_first")
    R = len(tau)
    pb.tau_q = np.array(tau, np.int32)
    pb.xi_q = np.array([1024, 512, 200, 64][:R - 1] + [64], np.int32)
    pb.rc_masks = np.array(policies, np.uint32)
    pb.eta_q = 1024 if N % 3 == 0 else 0
    o = Oracle(pb)
    _, best, index, _, _ = (o.search_pconfs_refined if objective == "refine" else o.search_pconfs_exact)(0, 1, threads=NTHREADS)
    hp = hap.hap_problem_create(pb, flags=hap.OPT_REFINE if objective == "refine" else hap.OPT_EXACT)
    hap.hap_enumerate(hp)
    if best < INF:
        plan, st = hap.hap_search_best(hp)
        assert (plan["index"], plan["T_iter"]) == (index, best)
        want = (o.eval_index_refined if objective == "refine" else o.eval_index_exact)(index)
        assert plan["n"] == want["n"] and plan["r"] == want["r"] and st["n_evaluated"] + st["n_pruned"] == hp.n_cand
    else:
        with pytest.raises(hap.HapError):
            hap.hap_search_best(hp)
    hap.hap_problem_destroy(hp)


@pytest.mark.parametrize("nodes,N,tau,policies,kinds", [CASES[2], CASES[4], ((2, 1, 1), 24, (0, 1024), (1, 3, 2), "uniform")])
def test_ranges_of_a_pass_whose_items_take_one_policy(nodes, N, tau, policies, kinds):
    """Ranges that begin and end between the policies of a mapping, and inside a configuration, against the oracle."""
    import paper_2609_39350_b200 as hap
    pb = problems.random_small(7 + N, N=N, T=len(nodes), nodes_per_type=nodes, node_size=2, window=True, first_dense=kinds == "dense_first")
    R = len(tau)
    pb.tau_q = np.array(tau, np.int32)
    pb.xi_q = np.array([1024, 512, 200, 64][:R - 1] + [64], np.int32)
    pb.rc_masks = np.array(policies, np.uint32)
    o = Oracle(pb)
    _, _, _, costs, _ = o.search_pconfs(0, 1, threads=NTHREADS, want_costs=True)
    hp = hap.hap_problem_create(pb)
    hap.hap_enumerate(hp)
    cuts = sorted(np.random.default_rng(N).integers(1, hp.n_cand, 5).tolist())
    for a, b in zip([0] + cuts, cuts + [hp.n_cand]):
        if a < b:
            assert np.array_equal(hap.hap_pipeline_dp(hp, a, b - a)["cost"].cpu().numpy(), costs[a:b]), (a, b)
    hap.hap_problem_destroy(hp)


@pytest.mark.parametrize("tau,policies", [((0, 1024), (3,)), ((0, 307, 1024), (1, 3, 7)), ((0, 1024, 2048), (7, 1))])
def test_items_of_several_configurations(tau, policies):
    """64 devices: classes of one or two parts share blocks, the last block of a class with fewer configurations; whole passes, ranges
    that begin inside a block's configurations, searches, and the fp64 pass."""
    import paper_2609_39350_b200 as hap
    pb = problems.mixtral()
    R = len(tau)
    pb.tau_q = np.array(tau, np.int32)
    pb.xi_q = np.array([1024, 400, 64][:R - 1] + [64], np.int32)
    pb.rc_masks = np.array(policies, np.uint32)
    o = Oracle(pb)
    _, best, index, costs, _ = o.search_pconfs(0, 1, threads=NTHREADS, want_costs=True)
    hp = hap.hap_problem_create(pb)
    hap.hap_enumerate(hp)
    assert np.array_equal(hap.hap_pipeline_dp(hp, 0, hp.n_cand)["cost"].cpu().numpy(), costs)
    for a in np.random.default_rng(R).integers(0, hp.n_cand - 5000, 4).tolist():
        assert np.array_equal(hap.hap_pipeline_dp(hp, a, 4999)["cost"].cpu().numpy(), costs[a:a + 4999]), a
    plan, _ = hap.hap_search_best(hp)
    assert (plan["index"], plan["T_iter"]) == (index, best)
    whole = hap.hap_pipeline_dp(hp, 0, hp.n_cand)["bottleneck"].cpu().numpy()
    f64 = hap.hap_pipeline_dp_f64(hp, 0, hp.n_cand)["bottleneck"].cpu().numpy()
    fin = whole < INF
    # a stage cost is a sum of numbers rounded to whole nanoseconds: forward and backward of at most N layers (half each), the repeated
    # forward of at most twice that, its floor, three transfers and ends
    assert np.array_equal(np.isfinite(f64), fin) and np.max(np.abs(f64[fin] - whole[fin])) <= 2 * pb.N + 4
    hap.hap_problem_destroy(hp)


@pytest.mark.parametrize("tau,policies", [((0, 1024), (3,)), ((0, 307, 1024), (1, 3, 7)), ((0, 1024, 2048), (7, 1))])
def test_costs_of_items_of_several_configurations(tau, policies):
    """As above with a dense first layer, and the unrounded costs, within 1e-9 relative of the fp64 oracle: sums, synchronisation and optimizer
    terms of every configuration of a block.  (That these calls take the grouped form: test_calls_that_share_blocks_between_configurations.)"""
    import paper_2609_39350_b200 as hap
    pb = problems.mixtral()
    R = len(tau)
    pb.kind[0] = 0
    pb.tau_q = np.array(tau, np.int32)
    pb.xi_q = np.array([1024, 400, 64][:R - 1] + [64], np.int32)
    pb.rc_masks = np.array(policies, np.uint32)
    o = Oracle(pb)
    _, best, index, costs, _ = o.search_pconfs(0, 1, threads=NTHREADS, want_costs=True)
    _, costs_f, bn_f, _ = o.search_pconfs_f64(0, 1, threads=NTHREADS)
    hp = hap.hap_problem_create(pb)
    hap.hap_enumerate(hp)
    assert np.array_equal(hap.hap_pipeline_dp(hp, 0, hp.n_cand)["cost"].cpu().numpy(), costs)
    plan, _ = hap.hap_search_best(hp)
    assert (plan["index"], plan["T_iter"]) == (index, best)
    got = {k: v.cpu().numpy() for k, v in hap.hap_pipeline_dp_f64(hp, 0, hp.n_cand).items()}
    for key, want in (("cost", costs_f), ("bottleneck", bn_f)):
        fin = np.isfinite(want)
        assert fin.any() and np.array_equal(fin, np.isfinite(got[key])), key
        assert np.max(np.abs(got[key][fin] - want[fin]) / want[fin]) <= 1e-9, key
    plan = hap.hap_search_range_f64(hp, 0, hp.n_cand)
    two = np.sort(costs_f[np.isfinite(costs_f)])[:2]
    assert plan["T_iter_f64"] == pytest.approx(two[0], rel=1e-9)
    assert plan["index"] == int(np.argmin(costs_f)) or two[1] - two[0] <= 1e-9 * two[0]
    hap.hap_problem_destroy(hp)


def test_searches_of_several_waves_with_three_levels():
    """256 devices, three levels combined into rows, one policy: some 13,000 items, of which two fifths are more than two waves, so that every
    search takes the kernels of four blocks an SM -- unpruned, in the order of the bounds, listing for refinement, unrounded."""
    import paper_2609_39350_b200 as hap
    pb = problems.dsv2()
    pb.tau_q = np.array((0, 1024, 2048), np.int32)
    pb.xi_q = np.array((1024, 400, 64), np.int32)
    pb.rc_masks = np.array((7,), np.uint32)
    o = Oracle(pb)
    _, best, index, _, _ = o.search_pconfs(0, 1, threads=NTHREADS, want_costs=True)
    for prune in (0, 1):
        hp = hap.hap_problem_create(pb, prune=prune)
        hap.hap_enumerate(hp)
        plan, st = hap.hap_search_best(hp)
        assert (plan["index"], plan["T_iter"]) == (index, best), prune
        want, _, _ = o.eval_index(index)
        assert plan["n"] == want["n"] and plan["r"] == want["r"] and st["n_evaluated"] + st["n_pruned"] == hp.n_cand
        if not prune:
            costs = hap.hap_pipeline_dp_f64(hp, 0, hp.n_cand)["cost"].cpu().numpy()
            got = hap.hap_search_range_f64(hp, 0, hp.n_cand)
            assert (got["index"], got["T_iter_f64"]) == (int(np.argmin(costs)), float(costs.min()))
            assert got["T_iter_f64"] == pytest.approx(o.eval_index_f64(got["index"])["T_iter"], rel=1e-9)
        hap.hap_problem_destroy(hp)
    for flag in (hap.OPT_REFINE, hap.OPT_EXACT):               # against one warp per candidate
        plans = []
        for more in (0, hap.OPT_NO_TRIE):
            hp = hap.hap_problem_create(pb, flags=flag | more)
            hap.hap_enumerate(hp)
            plan, _ = hap.hap_search_best(hp)
            plans.append((plan["index"], plan["T_iter"], plan["n"], plan["r"]))
            hap.hap_problem_destroy(hp)
        assert plans[0] == plans[1], flag
