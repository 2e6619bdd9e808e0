"""A device with little memory left: passes that have no room for the trees' records run without them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gen import problems  # noqa: E402


def test_a_pass_without_room_for_the_records():
    import paper_2609_39350_b200 as hap
    pb = problems.stress()
    pb.node_type = np.repeat(np.arange(4), [72, 27, 16, 13]).astype(np.int32)      # mixed stages: the records take 100 MB
    hp = hap.hap_problem_create(pb)
    _, n = hap.hap_enumerate(hp)
    want = hap.hap_pipeline_dp(hp, 0, n)["cost"].clone()
    best = hap.hap_search_best(hp)[0]
    hap.hap_problem_destroy(hp)
    hp = hap.hap_problem_create(pb, flags=hap.OPT_NO_TRIE)                         # (its kernels are loaded before memory is short)
    hap.hap_enumerate(hp)
    out = hap.hap_pipeline_dp(hp, 0, n)
    hap.hap_search_best(hp)
    assert torch.equal(out["cost"], want)
    hap.hap_problem_destroy(hp)
    out["cost"].zero_()
    torch.cuda.synchronize()
    hap.hap_release_cached_memory()
    torch.cuda.empty_cache()
    hold = []
    try:
        leave = 96 << 20                                                           # a pass without trees takes 12 + 48 MB
        while torch.cuda.mem_get_info()[0] - (1 << 30) >= leave:
            hold.append(torch.empty(1 << 30, dtype=torch.uint8, device="cuda"))
        rest = torch.cuda.mem_get_info()[0] - leave
        if rest > 10 << 20:                                                        # (the allocator takes smaller ones from 20 MB pieces)
            hold.append(torch.empty(rest, dtype=torch.uint8, device="cuda"))
        hp = hap.hap_problem_create(pb)
        assert hap.hap_enumerate(hp)[1] == n
        hap.hap_pipeline_dp(hp, 0, n, out=out)
        torch.cuda.synchronize()
        assert torch.equal(out["cost"], want)
        plan = hap.hap_search_best(hp)[0]
        assert (plan["index"], plan["T_iter"], plan["n"]) == (best["index"], best["T_iter"], best["n"])
        hap.hap_problem_destroy(hp)
    finally:
        hold.clear()
        hap.hap_release_cached_memory()
        torch.cuda.empty_cache()
