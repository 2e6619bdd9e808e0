"""The joint recurrence at the edges of its bit words (64 and 128 end layers a level; beyond them the form with a value per
end layer), with a dense first layer and with levels that are not combined into rows, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gen import problems  # noqa: E402
from oracle import Oracle  # noqa: E402


@pytest.mark.parametrize("nodes,N,window,tau,dense_first", [
    ((2, 2), 8, True, (0, 1024), False),              # as many layers as stages; few states: a value per end layer
    ((1, 1, 1, 1), 71, False, (0, 1024), False),      # 64 end layers at eight stages: one word, the last bit of it
    ((1, 1, 1, 1), 72, False, (0, 1024), False),      # 65: two words
    ((2, 2, 2, 2), 48, True, (0, 307, 1024), True),
    ((2, 1, 1), 130, False, (0, 1024), True),
    ((1, 1, 1, 1), 150, False, (0, 1024), False),     # more than two words
    ((2, 2, 2, 2), 33, True, (0, 500), False),
])
def test_joint_bottleneck_words(nodes, N, window, tau, dense_first):
    import paper_2609_39350_b200 as hap
    pb = problems.random_small(7 * N, N=N, T=len(nodes), nodes_per_type=nodes, node_size=2, window=window, first_dense=dense_first)
    pb.cap_eff[:] = pb.cap_eff * max(1, N // 8)    # (some policies fit, some do not)
    pb.tau_q = np.array(tau, np.int32)
    pb.xi_q = np.array([1024, 512, 64][-len(tau):], np.int32)
    pb.rc_masks = np.array([(1 << len(tau)) - 1, 1], np.uint32)
    o = Oracle(pb)
    hp = hap.hap_problem_create(pb)
    hap.hap_enumerate(hp)
    got = hap.hap_joint_bottleneck(hp).cpu().numpy()
    seen = 0
    for p in np.random.default_rng(N).permutation(o.n_pconf).tolist():
        for rc in range(2):
            if got[p, rc] == -1 or seen >= 60 or (seen >= 40 and o.pconfs[p]["PP"] < 8):
                continue
            c2, _, coef, _ = o.layer_costs(p)
            assert got[p, rc] == o.joint_bottleneck(p, int(pb.rc_masks[rc]), c2, coef), (p, rc)
            seen += 1
    assert seen > 0
    hap.hap_problem_destroy(hp)


@pytest.mark.parametrize("nodes,N,window,tau,dense_first", [
    ((2, 1, 1), 151, False, (0, 1024), True),         # 20,385 cells: every class in the form with a value per end layer
    ((2, 1, 1), 152, False, (0, 1024), True),         # 20,520: the classes of few cells beside the large one, in bits where they fit
    ((2, 2, 2, 2), 130, False, (0, 1024), True),      # two words, a dense first layer
])
def test_joint_bottleneck_forms(nodes, N, window, tau, dense_first):
    """Both sides of the line between the forms, which one class draws for all."""
    test_joint_bottleneck_words(nodes, N, window, tau, dense_first)


@pytest.mark.parametrize("nodes,N", [((1, 1, 1, 1), 131),      # at most 64 end layers a level, 71 with what lengths move down by: two words
                                     ((2, 1, 1), 226),         # 91 and 133: three words
                                     ((2, 2, 2, 2), 119)])     # eight and sixteen stages, 60 / 65 and 64 / 67
def test_joint_bottleneck_levels_that_begin_higher(nodes, N):
    """A level whose first end layer lies further up than the shortest stage of a type: its lengths are summed up below it."""
    test_joint_bottleneck_words(nodes, N, True, (0, 1024), False)


@pytest.mark.parametrize("nodes,N", [((1, 1, 1, 1), 226),      # eight stages, 135: three words
                                     ((2, 1, 1), 226)])        # four stages in three words would be 8,136 cells: a value per end layer, beside eight in bits
def test_joint_bottleneck_three_words(nodes, N):
    """Classes whose levels take three words, on both sides of the line between the forms."""
    test_joint_bottleneck_words(nodes, N, True, (0, 1024), False)
    test_joint_bottleneck_words(nodes, N, True, (0, 307, 1024), False)
