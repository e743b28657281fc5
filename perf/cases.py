"""The work a user of this library has it do, as cases that can be timed and compared.

listed() is the work at fixed sizes, draw() gives more of the same ranges.  A case is one call (or, for the
captured decode step, one replay) through the package's public entry points, on inputs made on the device from a
seed: bf16 caches of standard-normal keys and values (some with four key channels per head scaled by 8, as the
ragged batch of the workload generator has them), the generator's step layouts and signals, its budgets and head
shapes (8 query / 2 KV heads of 64, 32 / 8 and 40 / 8 of 128, and other group sizes the decode takes).

Kinds: "compress" (one pruning boundary per trajectory: saliency, priorities, selection, compaction -- out of
place, in place, or from a cache in pinned host memory), "score" (the saliency stage alone, long Observation
windows), "select" (the selection from saliency rows, with or without SnapKV-style pooling), "signals" (step
signals from evidence cues), "decode" (attention reads of a compacted cache, with or without accumulated
attention, all layers in one call or one call per layer in a captured decode step).
"""
import math
import random

import numpy as np
import torch

from paper_2609_22158_gb300 import binding as B
from paper_2609_22158_gb300 import cues as C
from paper_2609_22158_gb300 import workload as wl

DEV = "cuda"
N_PROMPT = 16  # protected prompt slots of every generated layout


# ------------------------------------------------------------------------------------------------ the cases
def _compress(name, L, Hq, Hkv, d, t_lo, W, n_steps, num=0, den=1, count=0, n_traj=1, t_hi=0, t_seed=0, outliers=0,
              in_place=False, host=False, lse=False, outputs="rows"):
    """num / den: a ratio budget, else count tokens; n_traj > 1: lengths uniform in [t_lo, t_hi] (drawn from t_seed);
    outputs: "rows" (the compacted cache and its metadata), "priority" (also P and T per token), "full" (also the
    per-step statistics)."""
    c = dict(kind="compress", L=L, Hq=Hq, Hkv=Hkv, d=d, t_lo=t_lo, t_hi=t_hi or t_lo, t_seed=t_seed, n_traj=n_traj,
             W=W, n_steps=n_steps, num=num, den=den, count=count, outliers=outliers, in_place=in_place, host=host,
             lse=lse, outputs=outputs)
    return dict(c, name=name) if name else c


def _score(name, n_layers, Hq, Hkv, d, T, W, lse=False, outliers=0):
    c = dict(kind="score", n_layers=n_layers, Hq=Hq, Hkv=Hkv, d=d, T=T, W=W, lse=lse, outliers=outliers)
    return dict(c, name=name) if name else c


def _select(name, rows, T, n_steps, pool, pool_mode, num, den):
    c = dict(kind="select", rows=rows, T=T, n_steps=n_steps, pool=pool, pool_mode=pool_mode, num=num, den=den)
    return dict(c, name=name) if name else c


def _signals(name, n_steps, k0):
    c = dict(kind="signals", n_steps=n_steps, k0=k0)
    return dict(c, name=name) if name else c


def _decode(name, L, Hq, Hkv, d, n, cap, h2o=False, per_layer=False, outliers=0):
    """n retained rows (read on the device, as after a compaction) of caches that hold cap rows."""
    c = dict(kind="decode", L=L, Hq=Hq, Hkv=Hkv, d=d, n=n, cap=cap, h2o=h2o, per_layer=per_layer, outliers=outliers)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the first boundaries of a short episode on a small model: latency and launches
        _compress("compress_short", 1, 8, 2, 64, 2048, 32, 8, num=1, den=4, outputs="full"),
        # one long trajectory of a 32-layer model at a 10% budget, the benchmark's workload
        _compress("compress_32k", 32, 32, 8, 128, 32768, 64, 40, num=1, den=10, outputs="priority"),
        # a serving batch of ragged trajectories compressed in one call
        _compress("compress_ragged", 32, 32, 8, 128, 8192, 64, 40, num=1, den=10, n_traj=16, t_hi=32768, t_seed=2,
                  outliers=4, outputs="rows"),
        # a long horizon on a 64-layer model with 5 query heads per KV head and a fixed budget: the largest call
        _compress("compress_64k", 64, 40, 8, 128, 65536, 128, 120, count=4096, outputs="full"),
        # one boundary of the incremental loop: the carried 8192-token cache plus one new step, in place
        _compress("compress_in_place", 32, 32, 8, 128, 8911, 64, 30, count=8192, in_place=True),
        # a cache kept in pinned host memory, compressed as it is fetched
        _compress("compress_from_host", 32, 32, 8, 128, 16384, 64, 40, num=1, den=10, host=True),
        # saliency from the whole last Observation, as collected during its prefill
        _score("score_observation", 3, 32, 8, 128, 32768, 2048),
        # selection from a caller's own saliency rows with the SnapKV-style estimator
        _select("select_pooled", 24, 32768, 40, 7, B.POOL_MAX, 1, 10),
        # the newest step's signals from its evidence cues, late in a long episode
        _signals("signals_120_steps", 120, 119),
        # one decoded token's attention over all layers of a compacted cache
        _decode("decode_32_layers", 32, 32, 8, 128, 8272, 8911, outliers=4),
        # the same token as an agent's model runs it: a call per layer, captured once as a graph
        _decode("decode_per_layer", 32, 32, 8, 128, 8272, 8911, per_layer=True, outliers=4),
        # decoding while accumulated attention is collected as the next boundary's saliency, 5 heads per KV head
        _decode("decode_h2o", 64, 40, 8, 128, 4240, 4999, h2o=True, outliers=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compress", "compress", "compress", "score", "select", "signals", "decode", "decode", "decode"])
    if kind == "compress":
        form = rng.choice(["plain", "plain", "batch", "in_place", "host", "lse"])
        if form == "host":
            L, (Hq, Hkv, d) = rng.choice([4, 16, 32]), rng.choice([(8, 2, 64), (32, 8, 128)])
            T = _log_int(rng, 1024, 16384)
        elif form == "batch":
            L, (Hq, Hkv, d) = rng.choice([4, 16]), rng.choice([(32, 8, 128), (40, 8, 128)])
            T = _log_int(rng, 1500, 12000)
        elif form == "in_place":
            L, (Hq, Hkv, d) = rng.choice([4, 32]), rng.choice([(32, 8, 128), (16, 8, 64)])
            T = _log_int(rng, 2500, 20000)
        else:
            L, (Hq, Hkv, d) = rng.choice([1, 8, 32]), rng.choice([(8, 2, 64), (32, 8, 128), (40, 8, 128)])
            T = _log_int(rng, 1000, 65536)
        W = rng.choice([16, 32, 57, 64, 128])
        n_steps = rng.randint(4, max(5, min(120, T // 250)))
        kw = dict(outliers=rng.choice([0, 4]), outputs=rng.choice(["rows", "priority", "full"]))
        if form == "in_place":
            kw.update(in_place=True, count=T - rng.randint(200, min(2000, T // 3)) - W)
        else:
            kw.update(num=rng.choice([1, 1, 2, 5]), den=rng.choice([10, 20]))
        if form == "batch":
            kw.update(n_traj=rng.randint(2, 16), t_hi=2 * T, t_seed=rng.randint(0, 999))
        kw.update(host=form == "host", lse=form == "lse")
        return _compress("", L, Hq, Hkv, d, T, W, n_steps, **kw)
    if kind == "score":
        Hq, Hkv, d = rng.choice([(8, 2, 64), (32, 8, 128), (40, 8, 128)])
        return _score("", rng.choice([1, 3]), Hq, Hkv, d, _log_int(rng, 4500, 32768 * 32 // max(32, Hq)),
                      rng.choice([200, 512, 1000, 2048]), lse=rng.random() < 0.3, outliers=rng.choice([0, 4]))
    if kind == "select":
        return _select("", rng.choice([2, 6, 24]), _log_int(rng, 600, 131072), rng.randint(4, 120),
                       rng.choice([1, 1, 5, 7, 13, 31]), rng.choice([B.POOL_MAX, B.POOL_AVG]), 1, rng.choice([4, 10, 20]))
    if kind == "signals":
        n = _log_int(rng, 6, 400)
        return _signals("", n, rng.choice([0, n - 1, n - 1]))
    Hq, Hkv, d = rng.choice([(8, 2, 64), (32, 8, 128), (32, 8, 128), (40, 8, 128), (16, 8, 64), (16, 16, 128), (64, 8, 128)])
    n = _log_int(rng, 100, 16384)
    return _decode("", rng.choice([1, 4, 32]), Hq, Hkv, d, n, n + rng.randint(0, 1500), h2o=rng.random() < 0.35,
                   per_layer=rng.random() < 0.35, outliers=rng.choice([0, 4]))


def _lengths(c):
    r = random.Random(c["t_seed"])
    return [c["t_lo"]] if c["n_traj"] == 1 else [r.randint(c["t_lo"], c["t_hi"]) for _ in range(c["n_traj"])]


def _kept(c, T):
    """Retained rows of one trajectory: the protected prompt and window, and the budget's share of the others."""
    n = T - N_PROMPT - c["W"]
    return N_PROMPT + c["W"] + min(n, max(1, n * c["num"] // c["den"]) if c["num"] else c["count"])


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(gen, *shape):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)


def _keys(gen, outliers, *shape):
    """Keys [..., rows, d]; with outliers, that many channels per head scaled by 8."""
    k = _randn(gen, *shape)
    if outliers:
        order = torch.rand((*shape[:-2], 1, shape[-1]), generator=gen, device=DEV).argsort(-1)
        k *= torch.where(order < outliers, 8.0, 1.0).to(torch.bfloat16)
    return k


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _row_lse(K, Q):
    """Natural-log causal log-sum-exp of every window query, [Hq, W] fp32: what a prefill attention reports."""
    Hkv, T, d = K.shape
    Hq, W, _ = Q.shape
    lim = (T - W + torch.arange(W, device=DEV))[:, None]
    hide = torch.arange(T, device=DEV)[None, :] > lim
    return torch.stack([torch.logsumexp((Q[g].float() @ K[g * Hkv // Hq].float().T / math.sqrt(d)).masked_fill(
        hide, float("-inf")), 1) for g in range(Hq)])


def _prepare_compress(c, seed):
    gen = _gen(seed)
    trajs, probs = [], []
    L, Hq, Hkv, d, W = c["L"], c["Hq"], c["Hkv"], c["d"], c["W"]
    reuse = torch.zeros((c["n_traj"], c["n_steps"]), dtype=torch.float32, device=DEV)
    for b, T in enumerate(_lengths(c)):
        tr = wl.custom(seed * 64 + b, L=L, Hq=Hq, Hkv=Hkv, d=d, T=T, W=W, n_steps=c["n_steps"], n_prompt=N_PROMPT)
        cap = _kept(c, T)
        K, V = _keys(gen, c["outliers"], L, Hkv, T, d), _randn(gen, L, Hkv, T, d)
        Ls = min(3, L)
        Q = [_randn(gen, Hq, W, d) for _ in range(Ls)]
        sal = None
        if c["host"]:
            sal = list(K[L - Ls:].clone())
            host = [torch.empty(x.shape, dtype=x.dtype, pin_memory=True) for x in (K, V)]
            K, V = host[0].copy_(K), host[1].copy_(V)
        Ko, Vo = (K, V) if c["in_place"] else (torch.zeros((L, Hkv, cap, d), dtype=torch.bfloat16, device=DEV) for _ in "kv")
        n = tr.n_steps
        steps = B.StepSignals(_dev(tr.valid), _dev(tr.gain), _dev(tr.red), _dev(tr.reuse), _dev(tr.obs_sim), reuse[b])
        out = B.SelectOutputs.allocate(T, n, cap, DEV, full=c["outputs"] == "full")
        if c["outputs"] == "priority":
            out.priority, out.token_sal = (torch.zeros(T, dtype=torch.float32, device=DEV) for _ in "pt")
        sid_out, pos_out = (torch.zeros(cap, dtype=torch.int32, device=DEV) for _ in "sp")
        budget = B.budget_ratio(c["num"], c["den"]) if c["num"] else B.budget_count(c["count"])
        lse = [_row_lse(K[L - Ls + i], Q[i]) for i in range(Ls)] if c["lse"] else None
        loc = dict(kv_location=B.STEPKV_MEM_HOST, K_sal=sal) if c["host"] else {}
        probs.append(B.Problem(list(K), list(V), Q, T, _dev(tr.step_id), _dev(tr.prot), steps, budget, list(Ko), list(Vo),
                               out, pos_in=_dev(tr.pos), step_id_out=sid_out, pos_out=pos_out, sal_lse=lse, **loc))
        trajs.append(dict(tr=tr, K=K, V=V, Ko=Ko, Vo=Vo, Q=Q, out=out, sid_out=sid_out, pos_out=pos_out))
    ws = torch.empty(B.stepkv_workspace_size(probs) + 512, dtype=torch.uint8, device=DEV)
    # what the user reads back: the caches whole, and the per-trajectory vectors (a batch's few of them)
    res = dict(K=[t["Ko"] for t in trajs], V=[t["Vo"] for t in trajs], kept_idx=[t["out"].kept_idx for t in trajs],
               reuse=reuse)
    if c["n_traj"] == 1:
        t, o = trajs[0], trajs[0]["out"]
        res.update(n_kept=o.n_kept, step_id=t["sid_out"], pos=t["pos_out"])
        if c["outputs"] != "rows":
            res.update(priority=o.priority, token_sal=o.token_sal)
        if c["outputs"] == "full":
            res.update(n_budget=o.n_budget, step_util=o.step_util, step_count=o.step_count, step_sal_sum=o.step_sal_sum,
                       step_sal_max=o.step_sal_max, step_kept=o.step_kept)
    return dict(kind="compress", probs=probs, trajs=trajs, params=B.Params(), ws=ws, status=B.new_status(), res=res)


def _prepare_score(c, seed):
    gen = _gen(seed)
    K = list(_keys(gen, c["outliers"], c["n_layers"], c["Hkv"], c["T"], c["d"]))
    Q = list(_randn(gen, c["n_layers"], c["Hq"], c["W"], c["d"]))
    need = B.load_library().stepkv_score_workspace_size(c["n_layers"], c["Hkv"], c["Hq"], c["T"], c["W"])
    return dict(kind="score", K=K, Q=Q, T=c["T"], lse=[_row_lse(k, q) for k, q in zip(K, Q)] if c["lse"] else None,
                sal=torch.zeros((c["n_layers"], c["Hkv"], c["T"]), dtype=torch.float32, device=DEV),
                ws=torch.empty(need + 512, dtype=torch.uint8, device=DEV), status=B.new_status())


def _prepare_select(c, seed):
    T = c["T"]
    # saliency rows as a window of queries leaves them: about one per token, log-normal over the tokens, a few
    # tokens far above the rest
    g = np.random.default_rng(seed)
    sal = np.exp(g.standard_normal((c["rows"], T), dtype=np.float32) * np.float32(0.4)) * np.exp(
        g.standard_normal(T, dtype=np.float32))
    tr = wl.custom(seed, L=1, Hq=8, Hkv=2, d=64, T=T, W=32, n_steps=c["n_steps"], n_prompt=N_PROMPT)
    n = tr.n_steps
    steps = B.StepSignals(_dev(tr.valid), _dev(tr.gain), _dev(tr.red), _dev(tr.reuse), _dev(tr.obs_sim),
                          torch.zeros(n, dtype=torch.float32, device=DEV))
    out = B.SelectOutputs.allocate(T, n, _kept(dict(c, W=32, count=0), T), DEV)
    need = B.load_library().stepkv_select_workspace_size(c["rows"], T, n)
    return dict(kind="select", sal=_dev(sal), step_id=_dev(tr.step_id), prot=_dev(tr.prot), steps=steps, out=out, tr=tr,
                params=B.Params(sal_pool=c["pool"], sal_pool_mode=c["pool_mode"]), budget=B.budget_ratio(c["num"], c["den"]),
                ws=torch.empty(need + 512, dtype=torch.uint8, device=DEV), status=B.new_status())


def _prepare_signals(c, seed):
    n = c["n_steps"]
    fields = wl.synthetic_cues(seed, n)
    ids, cnt = C.pack_cues(fields)
    return dict(kind="signals", fields=fields, cues=_dev(ids.view(np.int32)), cnt=_dev(cnt), k0=c["k0"], status=B.new_status(),
                gain=torch.zeros(n, dtype=torch.float32, device=DEV), red=torch.zeros(n, dtype=torch.float32, device=DEV),
                obs_sim=torch.zeros(n, dtype=torch.float32, device=DEV))


def _prepare_decode(c, seed):
    gen = _gen(seed)
    L, Hq, Hkv, d, cap = c["L"], c["Hq"], c["Hkv"], c["d"], c["cap"]
    K, V, q = _keys(gen, c["outliers"], L, Hkv, cap, d), _randn(gen, L, Hkv, cap, d), _randn(gen, L, Hq, d)
    out = torch.zeros((L, Hq, d), dtype=torch.float32, device=DEV)
    mass = torch.zeros((L, Hkv, cap), dtype=torch.float32, device=DEV) if c["h2o"] else None
    n = torch.tensor([c["n"]], dtype=torch.int32, device=DEV)
    lib = B.load_library()
    size = lib.stepkv_decode_h2o_workspace_size if c["h2o"] else lib.stepkv_decode_workspace_size
    ws = torch.empty(size(1 if c["per_layer"] else L, Hkv, Hq, d, cap) + 512, dtype=torch.uint8, device=DEV)
    status = B.new_status()

    def read(lo, hi):
        a = (list(q[lo:hi]), list(K[lo:hi]), list(V[lo:hi]), n)
        if c["h2o"]:
            B.stepkv_decode_h2o(*a, list(mass[lo:hi]), out=list(out[lo:hi]), ws=ws, status=status)
        else:
            B.stepkv_decode(*a, out=list(out[lo:hi]), ws=ws, status=status)

    graph = None
    if c["per_layer"]:  # the decode step of a model: one call per layer, captured once and replayed per token
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            read(0, 1)
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for layer in range(L):
                read(layer, layer + 1)
        out.zero_()
        if mass is not None:
            mass.zero_()
    args = (list(q), list(K), list(V), n)
    return dict(kind="decode", q=q, K=K, V=V, out=out, mass=mass, n=n, ws=ws, status=status, graph=graph, args=args,
                outs=list(out), masses=None if mass is None else list(mass))


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, int(seed))


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    if s["kind"] == "compress":
        B.stepkv_compress(s["probs"], s["params"], ws=s["ws"], status=s["status"])
        return dict(s["res"], status=s["status"])
    if s["kind"] == "score":
        B.stepkv_score(s["K"], s["Q"], s["T"], sal=s["sal"], ws=s["ws"], status=s["status"], lse=s["lse"])
        return dict(sal=s["sal"], status=s["status"])
    if s["kind"] == "select":
        o = B.stepkv_select(s["sal"], s["step_id"], s["prot"], s["steps"], s["params"], s["budget"], s["out"], ws=s["ws"],
                            status=s["status"])
        return dict(kept_idx=o.kept_idx, n_kept=o.n_kept, n_budget=o.n_budget, priority=o.priority, token_sal=o.token_sal,
                    step_util=o.step_util, step_count=o.step_count, step_sal_sum=o.step_sal_sum,
                    step_sal_max=o.step_sal_max, step_kept=o.step_kept, reuse=s["steps"].reuse_out, status=s["status"])
    if s["kind"] == "signals":
        B.stepkv_step_signals(s["cues"], s["cnt"], k0=s["k0"], gain=s["gain"], red=s["red"], obs_sim=s["obs_sim"],
                              status=s["status"])
        return dict(gain=s["gain"], red=s["red"], obs_sim=s["obs_sim"], status=s["status"])
    if s["graph"] is not None:
        s["graph"].replay()
    elif s["mass"] is not None:
        B.stepkv_decode_h2o(*s["args"], s["masses"], out=s["outs"], ws=s["ws"], status=s["status"])
    else:
        B.stepkv_decode(*s["args"], out=s["outs"], ws=s["ws"], status=s["status"])
    return dict(out=s["out"], status=s["status"]) if s["mass"] is None else dict(out=s["out"], mass=s["mass"], status=s["status"])


# ------------------------------------------------------------------------------------------------ what it takes
def work(c):
    if c["kind"] == "compress":
        total = flops = 0
        for T in _lengths(c):
            Ls = min(3, c["L"])
            # rows that have to move: every retained row, or in place at least the window, which lies beyond them
            rows = c["W"] if c["in_place"] else _kept(c, T)
            total += Ls * (c["Hkv"] * T + c["Hq"] * c["W"]) * c["d"] * 2          # keys and window queries
            total += 2 * 2 * c["L"] * c["Hkv"] * rows * c["d"] * 2                # K and V rows read and written
            total += 5 * T + 20 * _kept(c, T) + (8 * T if c["outputs"] != "rows" else 0)
            flops += 2 * Ls * c["Hq"] * c["W"] * T * c["d"]                       # one product of queries and keys
        return dict(bytes=total, flops=flops)
    if c["kind"] == "score":
        by = c["n_layers"] * ((c["Hkv"] * c["T"] + c["Hq"] * c["W"]) * c["d"] * 2 + 4 * c["Hkv"] * c["T"])
        return dict(bytes=by, flops=2 * c["n_layers"] * c["Hq"] * c["W"] * c["T"] * c["d"])
    if c["kind"] == "select":
        return dict(bytes=4 * c["rows"] * c["T"] + 13 * c["T"] + 4 * _kept(dict(c, W=32, count=0), c["T"]) + 36 * c["n_steps"],
                    flops=c["rows"] * c["T"])
    if c["kind"] == "signals":
        return dict(bytes=c["n_steps"] * (3 * 64 * 4 + 3 * 4 + 4) + 8 * (c["n_steps"] - c["k0"]), flops=0)
    by = c["L"] * (2 * c["Hkv"] * c["n"] * c["d"] * 2 + c["Hq"] * c["d"] * 6 + (8 * c["Hkv"] * c["n"] if c["h2o"] else 0))
    return dict(bytes=by, flops=4 * c["L"] * c["Hq"] * c["n"] * c["d"])


def tolerance(c):
    # About four times the largest relative error measured against exact() (32-bit sums in another order): priorities
    # and token saliency 1.7e-7, saliency rows 3.3e-7, decode outputs and masses 6.3e-7, step signals 2.6e-8.  A retained
    # set is equal but for ties within rounding of the last kept priority.
    rel = dict(compress=1e-6, select=1e-6, score=2e-6, decode=3e-6, signals=1e-7)[c["kind"]]
    return dict(rel=rel, differ=0.01) if c["kind"] in ("compress", "select") else dict(rel=rel)


# ------------------------------------------------------------------------------------------------ 64-bit values
def _saliency64(K, Q):
    """[Hkv, T] group-mean window attention of one layer."""
    Hkv, T, d = K.shape
    Hq, W, _ = Q.shape
    G = Hq // Hkv
    A = torch.zeros((Hkv, T), dtype=torch.float64, device=DEV)
    col = torch.arange(T, device=DEV)[None, :]
    for h in range(Hkv):
        k = K[h].double()
        rows = Q[h * G:(h + 1) * G].reshape(G * W, d).double()
        lim = (T - W + torch.arange(G * W, device=DEV) % W)[:, None]
        for r in range(0, G * W, 2048):
            x = (rows[r:r + 2048] @ k.T / math.sqrt(d)).masked_fill_(col > lim[r:r + 2048], float("-inf"))
            A[h] += torch.softmax(x, 1).sum(0)
        A[h] /= G
    return A


def _boundary64(tr, T_raw, params):
    """Eqs. 2-5 and the per-step statistics of one boundary from its raw token saliency."""
    f = lambda a: np.asarray(a, np.float64)
    prunable = tr.prot == 0
    reuse = f(tr.reuse) + np.minimum(1.0, params.eta * f(tr.obs_sim))
    reuse[-1] = 0.0
    r = f(tr.valid) + f(tr.gain) - params.lam * f(tr.red)
    S = np.clip(params.w_r * np.clip(r, params.r_min, params.r_max) + params.w_c * np.log1p(reuse), 0.0, params.s_max)
    th = T_raw / T_raw[prunable].max()
    P = np.where(prunable, params.alpha * th + params.beta * S[np.maximum(tr.step_id, 0)], -np.inf)
    sid, n = tr.step_id[prunable], tr.n_steps
    smax = np.zeros(n)
    np.maximum.at(smax, sid, th[prunable])
    return dict(reuse=reuse, priority=P, token_sal=th, step_util=S, step_sal_max=smax,
                step_sal_sum=np.bincount(sid, th[prunable], n))


def _exact_compress(c, s):
    got = []
    for t in s["trajs"]:
        Ls = len(t["Q"])
        T_raw = torch.cat([_saliency64(t["K"][c["L"] - Ls + i].to(DEV), t["Q"][i]) for i in range(Ls)]).mean(0)
        got.append(_boundary64(t["tr"], T_raw.cpu().numpy(), s["params"]))
    reuse = np.stack([g["reuse"] for g in got])
    return dict({k: v for k, v in got[0].items() if k in s["res"] and c["n_traj"] == 1}, reuse=reuse)


def _exact_select(c, s):
    x = s["sal"].double()
    h = c["pool"] // 2
    if h and c["pool_mode"] == B.POOL_MAX:
        x = torch.nn.functional.max_pool1d(x[:, None], c["pool"], 1, h)[:, 0]
    elif h:
        x = torch.nn.functional.avg_pool1d(x[:, None], c["pool"], 1, h, count_include_pad=False)[:, 0]
    return _boundary64(s["tr"], x.mean(0).cpu().numpy(), s["params"])


def _exact_signals(c, s):
    n, k0 = c["n_steps"], c["k0"]
    F = s["fields"]
    sim = lambda a, b: len(a & b) / len(a | b) if a | b else 0.0
    th_ob, act, obs = ([set(map(int, np.concatenate([F[k][i] for i in part]))) for k in range(n)]
                       for part in ((0, 2), (1,), (2,)))
    gain, red, osim = np.zeros(n), np.zeros(n), np.zeros(n)
    for k in range(k0, n):
        gain[k] = 1.0 - max([sim(th_ob[k], th_ob[u]) for u in range(k)], default=0.0)
        red[k] = max([sim(act[k], act[u]) for u in range(k)], default=0.0)
    osim[:n - 1] = [sim(obs[n - 1], obs[k]) for k in range(n - 1)]
    return dict(gain=gain, red=red, obs_sim=osim)


def _exact_decode(c, s):
    L, Hq, Hkv, d, n = c["L"], c["Hq"], c["Hkv"], c["d"], c["n"]
    G = Hq // Hkv
    out, mass = torch.zeros((L, Hq, d), dtype=torch.float64), torch.zeros((L, Hkv, c["cap"]), dtype=torch.float64)
    for l in range(L):
        p = torch.softmax(s["q"][l].double().view(Hkv, G, d) @ s["K"][l][:, :n].double().transpose(1, 2) / math.sqrt(d), -1)
        out[l] = (p @ s["V"][l][:, :n].double()).reshape(Hq, d).cpu()
        mass[l, :, :n] = p.mean(1).cpu()
    return dict(out=out, mass=mass) if c["h2o"] else dict(out=out)


def exact(case, seed):
    s = prepare(case, int(seed))
    if case["kind"] == "score":
        return dict(sal=torch.stack([_saliency64(k, q) for k, q in zip(s["K"], s["Q"])]))
    return globals()["_exact_" + case["kind"]](case, s)
