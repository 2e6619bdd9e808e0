"""Performance cases of the planner: what its users have it do, through the package's public entry points.

A case describes one planning problem (model shape, cluster inventory, search options) and what is asked about it:

  plan      plan once from host tables: create the problem, enumerate, search, release.  What a training launcher does
            whenever fresh profiles come in; everything starts from numpy arrays and ends with the plan on the host.
  search    search again on a problem that is kept (the calling program already holds the handle).
  pass      the cost and bottleneck of every candidate (optionally its partition and recomputation levels) left on the
            GPU, and the best of them: sensitivity studies, plots of the plan space, a rank's share of a sharded search.
  pass_f64  the same costs unrounded, in fp64.
  joint     the smallest bottleneck over all stage-type sequences of every configuration (bound on any mapping).
  costs     the layer-cost and stage-coefficient tables of every configuration.
  evaluate  closed-form (Appendix B) and simulated 1F1B latency of the plans of one configuration.

Model shapes and clusters are those of the repository's five configurations (8 to 1024 devices, 16 to 96 layers) and
what lies between them; tables are synthetic, as everywhere in this repository.
"""
import math

import numpy as np
import torch

import paper_2609_39350_b200 as hap

# the repository's model shapes and device types (see the generator of its five configurations)
_SHAPES = {
    "tiny": dict(layers=16, dense_first=0, seq=2048, hidden=1024, experts=8, topk=2, shared=0, ffn_dense=4096, ffn=4096,
                 heads=8, kv_heads=8, vocab=32000, types="400:80:400,200:40:400", nodes="1,1", node_size=4, micro="1,2,4,8",
                 uplink="25:25", zipf=1.2),
    "small": dict(layers=32, dense_first=0, seq=4096, hidden=2048, experts=64, topk=8, shared=0, ffn_dense=1024, ffn=1024,
                  heads=16, kv_heads=8, vocab=32000, types="400:80:900,300:64:400,150:32:200", nodes="2,1,1", node_size=8,
                  micro="1,2,4,8", uplink="50:50", zipf=1.2),
    "mixtral": dict(layers=32, dense_first=0, seq=4096, hidden=4096, experts=8, topk=2, shared=0, ffn_dense=14336, ffn=14336,
                    heads=32, kv_heads=8, vocab=32000, types="400:80:900,250:64:300", nodes="4,4", node_size=8,
                    micro="1,2,4,8", uplink="50:50", zipf=1.2),
    "dsv2": dict(layers=60, dense_first=1, seq=4096, hidden=5120, experts=160, topk=6, shared=2, ffn_dense=12288, ffn=1536,
                 heads=128, kv_heads=128, vocab=102400, types="400:80:900,300:64:600,200:48:400,150:32:200", nodes="12,8,8,4",
                 node_size=8, micro="1,2,4,8", uplink="25:50", zipf=1.4),
    "stress": dict(layers=96, dense_first=0, seq=8192, hidden=8192, experts=256, topk=8, shared=0, ffn_dense=2048, ffn=2048,
                   heads=64, kv_heads=8, vocab=128000, types="400:80:900,300:64:600,250:48:400,150:32:200",
                   nodes="64,32,16,16", node_size=8, micro="1,2,4", uplink="50:50", zipf=1.2),
}
_RACK = {"dsv2": 4, "stress": 32}
_BATCH = {"tiny": 64, "small": 256, "mixtral": 512, "dsv2": 1024, "stress": 2048}

# search options, in the form a case carries them: the load-balance window (1/1024, < 0 off) and the cap on enumerated
# mappings; recomputation levels as (activation factor, repeated forward fraction) in 1/1024 and the allowed levels of
# each policy; Pruning 3's eta (1/1024, 0 off); whether a search may skip candidates by its lower bound; the objective
# ("" = bottleneck-optimal partition, "exact" = optimum of the pipeline term); a profiled link-efficiency table or none
_OPTIONS = dict(delta_q=205, map_cap=2048, levels="1024:0,64:1024", policies="3", eta_q=0, prune=False, objective="", links=False,
                plans=False)


def _case(op, shape, name=None, **changes):
    c = dict(name=name) if name else {}
    c.update(op=op, shape=shape, **_SHAPES[shape], batch=_BATCH[shape], **_OPTIONS)
    if shape == "stress":
        c["policies"] = "1,3"
    c.update(changes)
    return c


def listed():
    return [
        # the smallest call: one plan for two nodes of four devices, all latency
        _case("plan", "tiny", "plan_8_devices", delta_q=-1, map_cap=1 << 40),
        # an ordinary replan with the paper's defaults (delta 0.2, eta 2), profiled link table, pruning allowed
        _case("plan", "mixtral", "plan_64_devices", eta_q=2048, links=True, prune=True),
        # the largest replan: 2.4 million candidates
        _case("plan", "stress", "plan_1024_devices"),
        # a scheduler that asks the same problem again (the handle is kept), pruning allowed
        _case("search", "stress", "search_1024_devices_pruned", prune=True),
        # every candidate's cost, partition and recomputation levels; first layer dense
        _case("pass", "dsv2", "pass_256_devices_plans", plans=True),
        # the benchmark's step
        _case("pass", "stress", "pass_1024_devices"),
        # unrounded costs; an odd layer count and uneven node counts: shares and windows that do not divide evenly
        _case("pass_f64", "small", "pass_f64_56_devices_uneven", layers=29, nodes="3,3,1", batch=448),
        # three recomputation levels, the middle one re-executing 30 % of the forward pass (selective recomputation)
        _case("pass", "mixtral", "pass_64_devices_selective", levels="1024:0,400:307,64:1024", policies="1,3,7"),
        # the exact optimum of the pipeline term
        _case("search", "dsv2", "search_256_devices_exact", objective="exact"),
        # the bound over all stage-type sequences
        _case("joint", "stress", "joint_1024_devices"),
        # the cost tables themselves (what a user inspects or feeds to another search)
        _case("costs", "stress", "costs_1024_devices"),
        # post-hoc latency of the best configuration's plans
        _case("evaluate", "small", "evaluate_32_devices"),
    ]


def draw(rng):
    """A case of the same ranges: any of the operations on a cluster of 8 to 1024 devices and a model of 12 to 96
    layers, odd and uneven counts among them."""
    while True:
        shape = rng.choice(list(_SHAPES))
        base = _SHAPES[shape]
        op = rng.choice(["plan", "plan", "search", "search", "pass", "pass", "pass_f64", "joint", "costs", "evaluate"])
        types = base["types"].split(",")
        nodes = [int(x) for x in base["nodes"].split(",")]
        # the whole inventory, or part of each type's nodes (never less than 60 %, so that the model still fits)
        if rng.random() < 0.7:
            nodes = [rng.randint(max(1, math.ceil(0.6 * n)), n) for n in nodes]
        else:
            nodes = [n + rng.choice([0, 0, 1, 2]) for n in nodes] if shape in ("tiny", "small", "mixtral") else nodes
        keep = len(types) if rng.random() < 0.75 else rng.randint(max(1, len(types) - 2), len(types))
        if keep < len(types):                            # fewer device types: the dropped ones' nodes go to the first type
            nodes = [nodes[0] + sum(nodes[keep:])] + nodes[1:keep]
            types = types[:keep]
        # large clusters grow by whole racks: degrees are powers of two, and a model that needs hundreds of devices does
        # not fit a cluster whose device count has few factors of two
        nodes[0] += -sum(nodes) % _RACK.get(shape, 1)
        layers = max(12, int(round(math.exp(rng.uniform(math.log(base["layers"] * 0.55), math.log(base["layers"]))))))
        devices = sum(nodes) * base["node_size"]
        c = _case(op, shape, layers=layers, types=",".join(types), nodes=",".join(map(str, nodes)), batch=devices * rng.choice([2, 4, 8]),
                  delta_q=rng.choice([205, 205, 205, 300, 150]), eta_q=rng.choice([0, 0, 2048]), links=rng.random() < 0.3,
                  prune=rng.random() < 0.5, plans=op == "pass" and rng.random() < 0.4)
        c["policies"] = rng.choice(["3", "3", "1,3"])
        if op in ("search", "pass") and shape != "stress" and rng.random() < 0.25:
            c["levels"], c["policies"] = "1024:0,%d:%d,64:1024" % (rng.randint(200, 700), rng.randint(100, 500)), rng.choice(["7", "1,3,7"])
        elif op == "search" and rng.random() < 0.25:
            c["objective"] = rng.choice(["exact", "refine"])
        if op != "search" and op != "plan":
            c["prune"] = False
        if op in ("joint", "costs", "evaluate"):
            c["eta_q"] = 0
        if c["batch"] * layers > 1 << 20:
            continue
        n_conf, n_cand, classes = _space(c)
        if op == "joint" and not any(cnt for _, _, _, cnt in classes):
            continue                                     # no configuration has stages of one device type each
        most = 2_410_320 if c["levels"] == _OPTIONS["levels"] else 150_000
        if n_conf >= 64 and n_cand <= most:
            return c


# ---- the planning problem of a case ------------------------------------------------------------------------------


def _ints(text):
    return [int(x) for x in text.split(",")]


def _pow2(most):
    return [1 << i for i in range(most.bit_length()) if 1 << i <= most]


class Planning:
    """The planner's inputs as host arrays, with the field names that hap_problem_create reads."""

    def __init__(self, c, seed):
        rng = np.random.RandomState(seed % (1 << 31))
        types = [[int(x) for x in t.split(":")] for t in c["types"].split(",")]      # TFLOP/s, GB, bytes/ns inside a node
        nodes = _ints(c["nodes"])
        T, N = len(types), c["layers"]
        f64 = lambda v: np.ascontiguousarray(v, np.float64)        # noqa: E731
        i32 = lambda v: np.ascontiguousarray(v, np.int32)          # noqa: E731
        i64 = lambda v: np.ascontiguousarray(v, np.int64)          # noqa: E731
        self.N, self.S, self.H, self.E, self.k, self.n_shared = N, c["seq"], c["hidden"], c["experts"], c["topk"], c["shared"]
        self.F_dense, self.F_exp, self.nq, self.nkv, self.V = c["ffn_dense"], c["ffn"], c["heads"], c["kv_heads"], c["vocab"]
        self.GB, self.beta = c["batch"], 2.0
        self.kind = np.ones(N, np.uint8)
        self.kind[:c["dense_first"]] = 0
        self.P = i64([t[0] * 1000 for t in types])
        self.C = i64([t[1] << 30 for t in types])
        self.node_size = i32([c["node_size"]] * T)
        self.bw_intra = f64([t[2] for t in types])
        self.node_type = i32(np.repeat(np.arange(T), nodes))
        lo, hi = _ints(c["uplink"].replace(":", ","))
        self.node_bw_inter = f64(lo + (hi - lo) * rng.random_sample(len(self.node_type)))
        tp, cp, mb = _pow2(min(8, c["node_size"])), [1, 2, 4, 8], _ints(c["micro"])
        self.tp_list, self.cp_list, self.mb_list, self.tpe_list = i32(tp), i32(cp), i32(mb), i32(tp)
        self.ep_list = i32([e for e in _pow2(self.E) if self.E % e == 0])
        self.pp_list = i32(_pow2(min(N, 32)))
        self.tp_max = c["node_size"]
        # profiled compute tables: time = flops / (TP CP) / (rate x efficiency); efficiencies U[0.4, 0.7] per type and layer
        eff = 0.4 + 0.3 * rng.random_sample((T, 1, 1, 1, N))
        rate = f64([t[0] * 1e3 for t in types]).reshape(T, 1, 1, 1)
        tok = f64(mb).reshape(1, 1, 1, -1) * self.S
        phi = ((0.97 ** np.arange(len(tp))).reshape(1, -1, 1, 1) * (0.98 ** np.arange(len(cp))).reshape(1, 1, -1, 1)
               * f64([{1: 0.85, 2: 0.92, 4: 0.96}.get(b, 1.0) for b in mb]).reshape(1, 1, 1, -1))
        split = f64(tp).reshape(1, -1, 1, 1) * f64(cp).reshape(1, 1, -1, 1)
        H, moe = float(self.H), self.kind.reshape(1, 1, 1, 1, N)
        attn = 2.0 * tok * H * (2.0 * H + 2.0 * (self.H * self.nkv // self.nq)) + 4.0 * tok * self.S * H
        ffn = 6.0 * tok[..., None] * H * np.where(moe == 1, self.F_exp, self.F_dense)
        more = np.where(moe == 1, self.n_shared * 6.0 * tok[..., None] * H * self.F_exp, 0.0)
        den = (split * rate * phi)[..., None] * eff
        self.tff, self.tdf = f64(ffn / den), f64((attn[..., None] + ffn + more) / den)
        self.tdb, self.tfb = 2.0 * self.tdf, 2.0 * self.tff
        self.tpost = f64(6.0 * tok * H * self.V / (split * rate * 0.5 * phi))
        self.tpre = np.zeros_like(self.tpost)
        # Zipf expert loads; what they are remains the same for every split of the experts
        load = (1.0 + np.arange(self.E)) ** -(c["zipf"] * (0.9 + 0.2 * rng.random_sample()))
        self.rho = f64([load.max() / load.mean()] * len(self.ep_list))
        self.eta = f64([0.95 - 0.05 * h for h in range(T)])
        self.croute = f64([2.0 * self.E / (0.3 * t[0] * 1e3) for t in types])
        self.copt = f64([4.8 / t[0] for t in types])
        self.kappa, self.alpha, self.chi, self.gamma = float(self.k), f64([2000.0, 8000.0, 12000.0]), 0.7, 0.5
        self.ovl_tp, self.ovl_cp, self.ovl_dp, self.capf = 1.0, 0.25, 0.5, 1.0
        self.act_coef = f64([34.0, 34.0 + 4.0 * self.k])
        self.cap_eff = i64([math.floor(t[1] * 2.0 ** 30 * 0.9 / (1.0 + 0.02 * h)) for h, t in enumerate(types)])
        levels = [_ints(v.replace(":", ",")) for v in c["levels"].split(",")]
        self.xi_q, self.tau_q = i32([v[0] for v in levels]), i32([v[1] for v in levels])
        self.rc_masks = np.ascontiguousarray(_ints(c["policies"]), np.uint32)
        self.delta_q, self.map_cap, self.eta_q = c["delta_q"], c["map_cap"], c["eta_q"]
        if c["links"]:                                    # link efficiency by message size, 64 KiB to 128 GiB
            self.fsize = f64(65536.0 * 8.0 ** np.arange(8))
            ramp = 0.35 + 0.65 * (1.0 + np.arange(8)) / 9.0
            self.feff = f64(np.clip(np.outer([0.97, 0.9, 0.75], ramp) + 0.03 * (rng.random_sample((3, 8)) - 0.5), 0.05, 1.0))


def _flags(c):
    return {"": 0, "exact": hap.OPT_EXACT, "refine": hap.OPT_REFINE}[c["objective"]]


def _open(c, seed):
    pb = Planning(c, seed)
    hp = hap.hap_problem_create(pb, prune=int(c["prune"]), flags=_flags(c))
    hap.hap_enumerate(hp)
    return hp


def prepare(case, seed):
    op = case["op"]
    if op == "plan":
        return dict(op=op, pb=Planning(case, seed), prune=int(case["prune"]), flags=_flags(case))
    hp = _open(case, seed)
    s = dict(op=op, hp=hp)
    if op == "pass":
        s["out"] = dict(cost=torch.empty(hp.n_cand, dtype=torch.int64, device="cuda"),
                        bottleneck=torch.empty(hp.n_cand, dtype=torch.int64, device="cuda"))
        if case["plans"]:
            s["out"].update(partition=torch.empty((hp.n_cand, hap.MAX_PP), dtype=torch.uint8, device="cuda"),
                            recompute=torch.empty((hp.n_cand, hap.MAX_PP), dtype=torch.uint8, device="cuda"))
    elif op == "costs":
        s["c2"] = torch.empty((hp.n_pconf, hp.T, hp.N, 2), dtype=torch.int64, device="cuda")
        s["coef"] = torch.empty((hp.n_pconf, hp.T, hap.NCOEF), dtype=torch.int64, device="cuda")
    elif op == "evaluate":
        best, _ = hap.hap_search_best(hp)
        rows = hap.hap_get_pconfs(hp)
        row = rows[np.searchsorted(rows["offset"], best["index"], side="right") - 1]
        s["first"], s["count"] = int(row["offset"]), int(row["nmap"]) * hp.n_rc
        s["plans"] = hap.hap_pipeline_dp(hp, s["first"], s["count"], partition=True)
    return s


def _numbers(p):
    """A plan as one array: index, degrees, policy, times, then layers, device types and level of every stage."""
    v = [p[k] for k in ("index", "PP", "TP", "CP", "DP", "EP", "TPE", "b", "M", "rc_mask", "T_iter", "bottleneck", "T_pipe", "T_sync",
                        "T_opt")]
    for k in ("n", "mask", "r"):
        v += p[k] + [0] * (hap.MAX_PP - len(p[k]))
    return np.array(v, np.int64)


def run(s):
    op = s["op"]
    if op == "plan":
        hp = hap.hap_problem_create(s["pb"], prune=s["prune"], flags=s["flags"])
        hap.hap_enumerate(hp)
        plan, _ = hap.hap_search_best(hp)
        hap.hap_problem_destroy(hp)
        return _numbers(plan)
    hp = s["hp"]
    if op == "search":
        plan, _ = hap.hap_search_best(hp)
        return _numbers(plan)
    if op == "pass":
        out = hap.hap_pipeline_dp(hp, 0, hp.n_cand, out=s["out"])
        return dict(out, best=hap.hap_argmin(hp, out["cost"]))
    if op == "pass_f64":
        return hap.hap_pipeline_dp_f64(hp, 0, hp.n_cand)
    if op == "joint":
        return hap.hap_joint_bottleneck(hp)
    if op == "costs":
        return hap.hap_eval_layer_costs(hp, c2=s["c2"], coef=s["coef"])
    if op == "evaluate":
        part, rec = s["plans"]["partition"], s["plans"]["recompute"]
        closed = hap.hap_eval_appendix_b(hp, s["first"], s["count"], part, rec, detail=True)
        sim = hap.hap_simulate_1f1b(hp, s["first"], s["count"], part, rec, detail=True)
        return dict(closed=closed["t_iter"], closed_detail=closed["detail"], sim=sim["t_iter"], sim_detail=sim["detail"])
    raise ValueError(op)


# ---- what a pass cannot do without ---------------------------------------------------------------------------------


def _space(c):
    """(configurations, candidates, [(PP, configurations, mappings, stages per type or None)]) of a case."""
    nodes, ns = _ints(c["nodes"]), c["node_size"]
    m = [n * ns for n in nodes]
    W, T, N, n_rc = sum(m), len(m), c["layers"], len(c["policies"].split(","))
    eps = [e for e in _pow2(c["experts"]) if c["experts"] % e == 0]
    classes, n_conf, n_cand = [], 0, 0
    for PP in _pow2(min(N, 32)):
        if W % PP:
            continue
        G, nmap, cnt = W // PP, math.factorial(T), None
        if all(x % G == 0 for x in m):
            cnt = [x // G for x in m]
            seqs = math.factorial(PP) // math.prod(math.factorial(x) for x in cnt)
            nmap = seqs if seqs <= c["map_cap"] else nmap
        conf = 0
        expert = [(e, t) for e in eps for t in _pow2(min(8, ns)) if G % e == 0 and G % (e * t) == 0]
        for TP in _pow2(min(8, ns)):
            if G % TP or c["heads"] % TP or c["kv_heads"] % TP:
                continue
            for CP in (1, 2, 4, 8):
                if G % (TP * CP) or c["seq"] % (2 * CP):
                    continue
                conf += len(expert) * sum(1 for b in _ints(c["micro"]) if c["batch"] % (G // (TP * CP) * b) == 0)
        classes.append((PP, conf, nmap, cnt))
        n_conf += conf
        n_cand += conf * nmap * n_rc
    return n_conf, n_cand, classes


def work(case):
    """Bytes: the profiled tables once and the results once.  Operations: Eq. 2 per (configuration, type, layer), and
    per candidate and stage the stage cost, the running maximum and sum (four); two per cell of the joint recurrence;
    two per stage and micro-batch of a simulated schedule."""
    n_conf, n_cand, classes = _space(case)
    T, N, n_rc = len(case["nodes"].split(",")), case["layers"], len(case["policies"].split(","))
    rows = T * len(_pow2(min(8, case["node_size"]))) * 4 * len(_ints(case["micro"]))
    tables = 8 * rows * (4 * N + 2)
    units = n_conf * T * N
    stages = sum(conf * nmap * n_rc * PP for PP, conf, nmap, _ in classes)
    op = case["op"]
    if op in ("plan", "search"):
        return dict(bytes=tables + 256, flops=14 * units + 4 * stages)
    if op == "pass":
        return dict(bytes=tables + n_cand * (80 if case["plans"] else 16), flops=14 * units + 4 * stages)
    if op == "pass_f64":
        return dict(bytes=tables + n_cand * 16, flops=14 * units + 4 * stages)
    if op == "joint":
        cells = sum(conf * n_rc * math.prod(x + 1 for x in cnt) * T * N for _, conf, _, cnt in classes if cnt)
        return dict(bytes=tables + 8 * n_conf * n_rc, flops=14 * units + 2 * cells)
    if op == "costs":
        return dict(bytes=tables + 16 * units + 8 * 21 * n_conf * T, flops=14 * units)
    # one configuration's plans: its row of the tables, the plans and seven numbers each (how many depends on the
    # winner: the largest class stands for them)
    count = max(nmap for _, _, nmap, _ in classes) * n_rc
    return dict(bytes=tables // max(1, rows // T) + count * (64 + 56), flops=14 * T * N + count * 2 * 8 * case["batch"])


def tolerance(case):
    # whole nanoseconds and bytes are the same bit for bit; unrounded fp64 sums agree to rounding
    return {"rel": 1e-9, "max": 1e-8} if case["op"] == "pass_f64" else "exact"
