"""Performance cases of the annealing library: whole calls through its public entry points.

Every case is one call (or the few calls that belong together) of a user's program: an anneal with its results read
back, a population resumed from the host, a batch, a served mix, the evaluation of given configurations, and one
resampling step on device buffers. Graph sizes, degrees, populations and schedules are those of the library's own
configurations, benchmark and tests; long schedules are shortened (fewer temperature steps over the same range of
inverse temperatures), so that every temperature regime keeps its share.

A case is a dict of plain values; ``kind`` says which call it is. Inputs come from the seed alone. Outputs are whole
numbers except the weight sums, inverse temperatures and free energies of the per-step records.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import sharded
from paper_2510_21105_gb300 import workloads as wl


def _anneal(name, graph, n, degree, R, K, S, beta_hi, **options):
    return dict(name=name, kind="anneal", graph=graph, n=n, degree=degree, R=R, K=K, S=S, beta_lo=0.1, beta_hi=beta_hi,
                **options)


def listed():
    return [
        # The smallest call in earnest: a quick look at a small graph, where launches and latency are all there is.
        _anneal("anneal_tiny", "random", 96, 14.0, 24, 12, 3, 2.0, nlm_period=4),
        # The 800-vertex random instance in full: mean degree 48, a small population, one replica block per few SMs.
        _anneal("anneal_gnp800", "random", 800, 47.9, 256, 100, 4, 3.0),
        # The headline workload, G63-shaped, with Houdayer moves; 200 of its 1000 temperature steps.
        _anneal("anneal_g63like", "random", 7000, 11.8454, 16384, 200, 10, 4.0, nlm_period=50),
        # The signed 100 x 100 torus with a large population; 80 of its 800 temperature steps.
        _anneal("anneal_torus100", "torus", 10000, 4.0, 32768, 80, 8, 3.5),
        # A mid-sized population on the G63-shaped graph under the ESS-adaptive schedule (it ends by itself).
        _anneal("anneal_adaptive", "random", 7000, 11.8454, 2048, 400, 4, 4.0, adaptive=1),
        # A dense graph (degree above 127: 16-bit fields) with block moves.
        _anneal("anneal_dense", "random", 500, 250.0, 1024, 40, 4, 1.0, nlm_period=10, nlm_kind=1),
        # A dumped population of a large planar graph put back, a few more steps, and the population read again.
        dict(name="resume_planar", kind="resume", graph="planar", n=18001, degree=6.0, R=1024, K=16, S=4, beta_lo=0.1,
             beta_hi=3.0),
        # A batch of mixed instances in one call, captured in a CUDA graph.
        dict(name="batch_mixed", kind="batch", count=9, K=30, S=4, beta_hi=3.0, use_graph=True),
        # A served mix: requests submitted to a running server, results collected as they finish.
        dict(name="served_mixed", kind="served", count=8, K=24, S=4, beta_hi=3.0, R_hi=8192),
        # Candidate configurations evaluated on the G63-shaped graph.
        dict(name="energies_g63like", kind="energies", graph="random", n=7000, degree=11.8454, R=600),
        # One resampling step on a caller's device buffers, as a latency-critical loop calls it.
        dict(name="resample_step", kind="resample", R=16384, dbeta=0.004, spread=60.0),
        # One resampling step of a rank that holds a shard of G63-shaped replicas: weights, plan, parents, row gather.
        dict(name="shard_step", kind="shard", R=16384, n=7008, dbeta=0.004, spread=60.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# No drawn anneal makes more spin-flip attempts than this (the listed ones reach 2.3e11 at the fast end).
MAX_ATTEMPTS = 3.0e10


def draw(rng):
    kind = rng.choice(["anneal"] * 6 + ["resume", "batch", "served", "energies", "resample", "shard"])
    if kind in ("anneal", "resume"):
        graph = rng.choice(["random", "random", "torus", "planar"])
        n = _log_int(rng, 90, 20000)
        if graph == "torus":
            n = max(9, int(round(math.sqrt(n)))) ** 2
        degree = 4.0 if graph == "torus" else 6.0 if graph == "planar" else round(
            math.exp(rng.uniform(math.log(3.0), math.log(min(60.0, n / 4)))), 3)
        if graph == "random" and rng.random() < 0.15:   # dense: degree above 127
            n = rng.randint(300, 700)
            degree = round(n * rng.uniform(0.45, 0.6), 3)
        S = rng.randint(1, 10)
        R = _log_int(rng, 17, 20000 if kind == "anneal" else 1500)
        K = max(4, min(rng.randint(10, 200), int(MAX_ATTEMPTS / (float(n) * R * S))))
        R = max(4, min(R, int(MAX_ATTEMPTS / (float(n) * K * S))))
        case = dict(kind=kind, graph=graph, n=n, degree=degree, R=R, K=K, S=S, beta_lo=round(rng.uniform(0.05, 0.3), 3),
                    beta_hi=round(rng.uniform(1.0, 4.0), 3))
        if kind == "anneal":
            extra = rng.choice(["none", "none", "houdayer", "block", "ess", "acceptance", "reheat"])
            if extra == "houdayer":
                case["nlm_period"] = rng.randint(5, 50)
            elif extra == "block":
                case.update(nlm_period=rng.randint(5, 50), nlm_kind=1, nlm_block=rng.randint(2, 64))
            elif extra == "ess":
                case["adaptive"] = 1
            elif extra == "acceptance":
                case["adaptive"] = 2
            elif extra == "reheat":
                case.update(reheat_after=rng.randint(3, 10), reheat_back=rng.randint(1, 5))
        return case
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 9), K=rng.randint(8, 30), S=rng.randint(1, 4),
                    beta_hi=round(rng.uniform(1.5, 4.0), 3), use_graph=rng.random() < 0.5)
    if kind == "served":
        return dict(kind="served", count=rng.randint(2, 8), K=rng.randint(8, 24), S=rng.randint(1, 4),
                    beta_hi=round(rng.uniform(1.5, 4.0), 3), R_hi=_log_int(rng, 1024, 8192))
    if kind == "energies":
        n = _log_int(rng, 90, 20000)
        return dict(kind="energies", graph="random", n=n, degree=round(rng.uniform(3.0, min(40.0, n / 4)), 3),
                    R=max(1, min(_log_int(rng, 1, 2000), int(6.0e6 / n))))
    if kind == "resample":
        return dict(kind="resample", R=_log_int(rng, 1000, 32768), dbeta=round(rng.uniform(0.0005, 0.02), 5),
                    spread=round(rng.uniform(5.0, 100.0), 2))
    return dict(kind="shard", R=2 ** rng.randint(10, 14), n=_log_int(rng, 90, 18000),
                dbeta=round(rng.uniform(0.0005, 0.02), 5), spread=round(rng.uniform(5.0, 100.0), 2))


def _graph(kind, n, degree, seed):
    if kind == "torus":
        return wl.torus(int(round(math.sqrt(n))), seed=seed)
    if kind == "planar":
        return wl.delaunay(n, seed=seed)
    # m distinct pairs, uniform: the generator's law, drawn as whole arrays
    m = int(round(n * degree / 2))
    rng = np.random.default_rng(seed)
    keys = np.zeros(0, np.int64)
    while len(keys) < m:
        a, b = rng.integers(0, n, size=(2, 2 * m + 16))
        keep = a != b
        keys = np.unique(np.concatenate([keys, np.minimum(a, b)[keep] * n + np.maximum(a, b)[keep]]))
        keys = keys if len(keys) <= m else rng.choice(keys, size=m, replace=False)
    return wl.from_edges(n, keys // n, keys % n, name=f"random{n}")


def _mix(count, seed, R_of):
    """Mixed instances as the benchmark draws them: N from 800 to 20,000, random / signed torus / planar."""
    rng = np.random.default_rng(seed)
    out = []
    for t in range(count):
        n = 800 + 19200 * ((t * 5) % count) // count + 533 * (t % 4) + t   # the sizes are the mix's, the graphs the seed's
        kind = ("random", "torus", "planar")[t % 3]
        out.append((_graph(kind, n, 12.0, int(rng.integers(1 << 30))), R_of(t)))
    return out


def _spins(rng, R, n):
    return (rng.integers(0, 2, size=(R, n), dtype=np.int8) * 2 - 1).astype(np.int8)


def _energies(case, seed):
    """Replica energies as a population has them in mid-anneal: whole numbers, normally distributed, on the device."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.randn(case["R"], generator=gen, device="cuda")
    return (-10000 + x * case["spread"]).round().to(torch.int32)


_OPTIONS = ("nlm_period", "nlm_kind", "nlm_block", "adaptive", "reheat_after", "reheat_back")


def prepare(case, seed):
    kind, st = case["kind"], dict(case=case, seed=seed)
    rng = np.random.default_rng(seed)
    if kind in ("anneal", "resume"):
        g = _graph(case["graph"], case["n"], case["degree"], seed)
        st["ann"] = B.Annealer.from_graph(g)
        st["opts"] = {k: case[k] for k in _OPTIONS if k in case}
        if case.get("adaptive"):
            st["betas"], st["opts"]["beta_max"] = None, case["beta_hi"]
        else:
            st["betas"] = wl.linear_betas(case["beta_lo"], case["beta_hi"], case["K"])
        if kind == "resume":
            st["spins"] = _spins(rng, case["R"], g.n)
    elif kind == "batch":
        inst = _mix(case["count"], seed, lambda t: (1024, 4096, 16384)[t % 3])
        st["anns"] = [B.Annealer.from_graph(g) for g, _ in inst]
        betas = wl.linear_betas(0.1, case["beta_hi"], case["K"])
        st["items"] = [(a, betas, R, case["S"], seed + t, case["K"], {})
                       for t, (a, (_, R)) in enumerate(zip(st["anns"], inst))]
    elif kind == "served":
        hi = math.log2(case["R_hi"])
        st["requests"] = _mix(case["count"], seed,
                              lambda t: int(round(2 ** (10 + (hi - 10) * ((t * 3) % case["count"] + 0.5) / case["count"]))))
        st["betas"] = wl.linear_betas(0.1, case["beta_hi"], case["K"])
        st["server"] = B.Server(64 << 30, n_streams=16, steps_per_tick=8)
    elif kind == "energies":
        g = _graph(case["graph"], case["n"], case["degree"], seed)
        st["ann"] = B.Annealer.from_graph(g)
        st["spins"] = _spins(rng, case["R"], g.n)
    elif kind == "resample":
        st["E"] = _energies(case, seed)
        st["parent"] = torch.empty(case["R"], dtype=torch.int32, device="cuda")
        st["counts"] = torch.empty(case["R"], dtype=torch.int32, device="cuda")
        st["stream"] = B.current_stream_handle()
    else:
        st["E"] = _energies(case, seed)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        bits = torch.randint(0, 2, (case["R"], case["n"]), generator=gen, device="cuda", dtype=torch.int8)
        st["spins"] = bits * 2 - 1
        st["shard"] = sharded.LibraryShard(case["R"], "cuda", stream=B.current_stream_handle())
    return st


def _records(ann, K):
    """Best record, best configuration and the per-step records (without their time stamps). An adaptive schedule ends
    by itself after some number of steps; its records are laid out over the K steps it may take."""
    cut, cfg, step, sweep = ann.best()
    out = dict(cut=cut, config=cfg, step=step, sweep=sweep)
    stats = ann.step_stats()
    for k, v in stats.items():
        if len(v) < K:
            stats[k] = np.zeros((K,) + v.shape[1:], v.dtype)
            stats[k][: len(v)] = v
    out.update({k: v for k, v in stats.items() if k not in ("t_ms", "T", "o")})
    out["T"] = stats["T"].view(np.int64)
    out["o"] = stats["o"].view(np.int32)
    return out


def run(st):
    case = st["case"]
    kind, seed = case["kind"], st["seed"]
    if kind == "anneal":
        st["ann"].anneal(st["betas"], case["R"], case["S"], seed, K=case["K"], **st["opts"])
        return _records(st["ann"], case["K"])
    if kind == "resume":
        ann, K = st["ann"], case["K"]
        ann.begin(st["betas"], case["R"], case["S"], seed)
        ann.set_state(st["spins"], K // 2)
        ann.run(K)
        spins, E = ann.state()
        return dict(spins=spins, E=E, **_records_of_best(ann))
    if kind == "batch":
        B.pa_batch_anneal(st["items"], use_graph=case["use_graph"])
        return [_records_of_best(a) for a in st["anns"]]
    if kind == "served":
        srv = st["server"]
        ids = [srv.submit(g, st["betas"], R, case["S"], seed + t) for t, (g, R) in enumerate(st["requests"])]
        got = {}
        while len(got) < len(ids):
            for rid in ids:
                if rid not in got and srv.poll(rid) not in (0, 1):
                    got[rid] = srv.result(rid)
                    srv.release(rid)
            time.sleep(0.0005)
        return [{k: got[r][k] for k in ("cut", "energy", "step", "sweep", "slot", "config")} for r in ids]
    if kind == "energies":
        E, cuts = st["ann"].energies(st["spins"])
        return dict(E=E, cuts=cuts)
    if kind == "resample":
        r = B.pa_resample_noalloc(st["E"].data_ptr(), case["R"], 1.0, 1.0 + case["dbeta"], seed, 3,
                                  st["parent"].data_ptr(), st["counts"].data_ptr(), stream=st["stream"])
        return dict(parent=st["parent"], counts=st["counts"], A=r["A"], T=r["T"], emin=r["emin"], o=r["o"])
    sh, R = st["shard"], case["R"]
    emin = sh.emin(st["E"])
    A, T = sh.partials(st["E"], emin, 1.0, 1.0 + case["dbeta"])
    o = sharded.resample_offset(seed, 3)
    plan = sharded.plan(1, 0, R, [A], [T], o)
    src, counts = sh.parents(R, o, plan)
    rows, erows = sh.gather(st["spins"], st["E"], src)
    return dict(emin=emin, A=plan["A"], T=plan["T"], src=src, counts=counts, rows=rows, E=erows)


def _records_of_best(ann):
    cut, cfg, step, sweep = ann.best()
    energy, _, _, slot = ann.best_record()
    return dict(cut=cut, config=cfg, step=step, sweep=sweep, energy=energy, slot=slot)


def exact(case, seed):
    """Weight sums and energies of the calls whose outputs follow from their inputs in one pass. An anneal's outputs
    follow from its random numbers step by step, so they have no such value."""
    kind = case["kind"]
    if kind == "energies":
        g = _graph(case["graph"], case["n"], case["degree"], seed)
        x = _spins(np.random.default_rng(seed), case["R"], g.n)
        i, j, w = g.edges()
        E = np.empty(case["R"], np.int64)
        for r in range(case["R"]):
            E[r] = int((w.astype(np.int64) * x[r, i] * x[r, j]).sum())
        return dict(E=E, cuts=(int(w.astype(np.int64).sum()) - E) // 2)
    if kind in ("resample", "shard"):
        E = _energies(case, seed).cpu().numpy().astype(np.float64)
        # the step from 1.0 to 1.0 + dbeta as doubles give it
        A = float(np.exp(-((1.0 + case["dbeta"]) - 1.0) * (E - E.min())).sum())
        if kind == "resample":
            return dict(parent=None, counts=None, A=A, T=None, emin=int(E.min()), o=None)
        return dict(emin=int(E.min()), A=A, T=None, src=None, counts=None, rows=None, E=None)
    return None


def work(case):
    """Bytes of the inputs and outputs, and the arithmetic a pass cannot do without: per attempt the sum over the
    neighbours, one random number and one decision (a multiply and a few logic operations each)."""
    kind = case["kind"]
    if kind in ("anneal", "resume"):
        n, R, K, S = case["n"], case["R"], case["K"], case["S"]
        steps = K - K // 2 if kind == "resume" else K
        attempts = float(n) * R * S * steps
        b = 2.0 * n * case["degree"] + 4 * n + 8 * K + n + K * (60 + 4 * S)
        if kind == "resume":
            b += 2.0 * R * n + 4 * R
        return dict(bytes=b, flops=attempts * (case["degree"] + 4))
    if kind in ("batch", "served"):
        Rs = ([(1024, 4096, 16384)[t % 3] for t in range(case["count"])] if kind == "batch" else
              [2 ** (10 + (math.log2(case["R_hi"]) - 10) * (t + 0.5) / case["count"]) for t in range(case["count"])])
        attempts = sum(10400.0 * r * case["K"] * case["S"] for r in Rs)
        return dict(bytes=case["count"] * (2.0 * 10400 * 8 + 10400 * 5 + 8 * case["K"]), flops=attempts * 12)
    if kind == "energies":
        n, R = case["n"], case["R"]
        return dict(bytes=2.0 * n * case["degree"] + 4 * n + float(R) * n + 12 * R, flops=R * n * case["degree"])
    if kind == "resample":
        return dict(bytes=12.0 * case["R"], flops=20.0 * case["R"])
    return dict(bytes=2.0 * case["R"] * case["n"] + 16.0 * case["R"], flops=20.0 * case["R"])
