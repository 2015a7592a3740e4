"""What a user of this library has it do, as cases that can be timed and compared.

A case is one pass of a selection job through the public entry points of ``paper_2510_02470_b200``: rows are sketched,
the sketch is frozen, the rows are scored against it and the best are kept (or one of these steps alone, where programs
call it alone). The kinds:

* ``path``    rows resident on the device, fed in calls of ``chunk`` rows (0: all in one call), as a training loop hands
              over its mini-batches; then freeze, score, select. ``sketches`` > 1 is the merged form of the sketch.
* ``factors`` the same for last-layer gradients given as their two factors (softmax - onehot, features).
* ``score``   new rows against a sketch that is kept (one sketch serves several scoring passes), class-balanced: scores
              per class and the per-class best.
* ``select``  the best of scores that the program has.
* ``host``    the whole path in one call on rows in pinned host memory.

Rows follow the repository's workloads: low-rank signal with noise and log-normal norms (``lowrank``), last-layer
gradients of a softmax head (``lastlayer``), and its device generators of long rows (``long``, ``model``).

A sketch is defined up to the signs and rotations of its rows, so the outputs are what follows from it uniquely: its row
norms (a program that keeps the sketch takes both), every row's score, and which rows are kept (as a mask over the
rows, which a sampler would use; rows whose scores tie to rounding may swap places in the ordered list).
"""
import math

import torch

import paper_2510_02470_b200 as sage
from paper_2510_02470_b200 import workloads

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # the selection step alone, on the scores of a 50,000-example training set
        {"name": "select_50k", "kind": "select", "N": 50000, "keep": 0.1},
        # a handful of short rows of odd length: what a smoke test or a toy model gives; launches and latency
        {"name": "path_tiny", "kind": "path", "rows": "lowrank", "N": 300, "D": 257, "ell": 8, "dtype": "f32", "chunk": 100,
         "sketches": 1, "keep": 0.25, "aligned": False},
        # a small model's gradients in 1,024-row calls (the smallest benchmark workload)
        {"name": "path_lowrank_1k", "kind": "path", "rows": "lowrank", "N": 4096, "D": 1024, "ell": 32, "dtype": "f32", "chunk": 1024,
         "sketches": 1, "keep": 0.1, "aligned": True},
        # bf16 rows of odd length packed without padding (no row starts on a 16-byte boundary), ragged calls, odd sketch size
        {"name": "path_ragged_bf16", "kind": "path", "rows": "lowrank", "N": 7777, "D": 3001, "ell": 47, "dtype": "bf16", "chunk": 1111,
         "sketches": 1, "keep": 0.3, "aligned": False},
        # last-layer gradients of a 10-class head for a whole training set: the usual way the method is run
        {"name": "path_lastlayer_10", "kind": "path", "rows": "lastlayer", "N": 50000, "D": 5130, "C": 10, "ell": 64, "dtype": "f32",
         "chunk": 1000, "sketches": 1, "keep": 0.1, "aligned": True},
        # the same job with 16 merged sketches
        {"name": "merged_lastlayer_10", "kind": "path", "rows": "lastlayer", "N": 50000, "D": 5130, "C": 10, "ell": 64, "dtype": "f32",
         "chunk": 0, "sketches": 16, "keep": 0.1, "aligned": True},
        # last-layer gradients of a 100-class head, bf16
        {"name": "path_lastlayer_100", "kind": "path", "rows": "lastlayer", "N": 20000, "D": 51300, "C": 100, "ell": 128, "dtype": "bf16",
         "chunk": 500, "sketches": 1, "keep": 0.1, "aligned": True},
        # the same head given as factors, so that no row is ever formed
        {"name": "factors_100", "kind": "factors", "N": 20000, "F": 512, "C": 100, "ell": 128, "dtype": "bf16", "chunk": 0, "keep": 0.1},
        # long rows, the largest sketch
        {"name": "path_long", "kind": "path", "rows": "long", "N": 8192, "D": 262144, "ell": 256, "dtype": "bf16", "chunk": 0,
         "sketches": 1, "keep": 0.1, "aligned": True},
        # full-model gradients of a CIFAR ResNet-18 in 512-row calls (the headline workload's rows)
        {"name": "path_model", "kind": "path", "rows": "model", "N": 640, "D": 11173962, "ell": 64, "dtype": "bf16", "chunk": 512,
         "sketches": 1, "keep": 0.1, "aligned": True},
        # re-scoring a training set against a kept sketch, class-balanced
        {"name": "score_classes", "kind": "score", "N": 50000, "D": 5130, "C": 10, "ell": 64, "dtype": "f32", "keep": 0.1, "aligned": True},
        # the whole path in one call on host rows
        {"name": "host_lowrank_1k", "kind": "host", "rows": "lowrank", "N": 4096, "D": 1024, "ell": 32, "dtype": "f32", "chunk": 0,
         "keep": 0.1, "aligned": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["path", "path", "path", "path", "merged", "factors", "score", "select", "host"])
    keep = round(rng.uniform(0.02, 0.4), 3)
    if kind == "select":
        return {"kind": "select", "N": _log_int(rng, 1000, 2000000), "keep": keep}
    dtype = rng.choice(["f32", "bf16"])
    eb = 4 if dtype == "f32" else 2
    if kind in ("factors", "score") or (kind != "host" and rng.random() < 0.4):
        C = _log_int(rng, 2, 120)
        D = C * _log_int(rng, 16, 640) + C
        rows = "lastlayer"
    else:
        C = 0
        D = _log_int(rng, 64, 1000000 if kind == "path" else 16000)
        rows = "lowrank"
    ell = _log_int(rng, 4, 256 if kind in ("path", "score") else 128)
    # the listed cases' largest pass, in rows: a shrink every ell + 1 rows costs at least ~0.15 ms of a chain, more with ell^2
    most = min(50000, int(1.2e9 / (D * eb)), int(0.15 * (ell + 1) / max(1.5e-4, 5.0e-8 * ell * ell)))
    if kind == "host":
        most = min(most, int(1.0e8 / (D * eb)))
    N = max(2 * ell, _log_int(rng, min(200, most), most))
    case = {"kind": "path" if kind == "merged" else kind, "N": N, "D": D, "ell": ell, "dtype": dtype, "keep": keep}
    if kind in ("path", "merged", "host"):
        case["rows"] = rows
        case["chunk"] = 0 if kind == "host" else rng.choice([0, min(N, _log_int(rng, 32, 2000))])
        case["sketches"] = rng.choice([2, 4, 8, 16]) if kind == "merged" else 1
    if kind == "factors":
        case.update({"F": (D - C) // C, "chunk": rng.choice([0, min(N, _log_int(rng, 64, 4000))])})
        del case["D"]
    else:
        case["aligned"] = rng.random() < 0.7
    if C:
        case["C"] = C
    return case


# ---- inputs --------------------------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rand(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _empty_rows(N, D, dtype, aligned):
    """N rows of D values, at a pitch of whole 16-byte units when aligned, packed otherwise."""
    ld = workloads.padded_pitch(D, 4 if dtype == torch.float32 else 2) if aligned else D
    return torch.zeros((N, ld), dtype=dtype, device="cuda")


def _lowrank(g, N, D, dtype, aligned, rank=16):
    """Rows s_i (c_i Q + 0.1 n_i), one in ten of them noise alone, as the small low-rank workload has them."""
    out = _empty_rows(N, D, dtype, aligned)
    Q = torch.linalg.qr(_rand(g, D, rank))[0].t().contiguous()
    step = max(1, (1 << 26) // D)
    for r0 in range(0, N, step):
        n = min(step, N - r0)
        c = _rand(g, n, rank) * (torch.rand((n, 1), generator=g, device="cuda") >= 0.1)
        x = _rand(g, n, D).mul_(0.1).addmm_(c, Q)
        out[r0:r0 + n, :D] = x * torch.exp(0.5 * _rand(g, n, 1))
    return out


def _head(g, N, C, F, flip=0.15):
    """The factors of the last-layer gradients of a softmax head over a Gaussian mixture with some labels moved."""
    mu = _rand(g, C, F)
    cls = torch.randint(C, (N,), generator=g, device="cuda")
    moved = torch.rand((N,), generator=g, device="cuda") < flip
    y = torch.where(moved, (cls + torch.randint(1, max(C, 2), (N,), generator=g, device="cuda")) % C, cls)
    h = torch.relu(mu[cls] + _rand(g, N, F))
    q = torch.softmax(h @ (torch.relu(mu) / math.sqrt(F)).t(), dim=1)
    q[torch.arange(N, device="cuda"), y] -= 1.0
    return q, h, y.to(torch.int32)


def _lastlayer(g, N, C, D, dtype, aligned):
    F = (D - C) // C
    q, h, y = _head(g, N, C, F)
    out = _empty_rows(N, D, dtype, aligned)
    step = max(1, (1 << 27) // D)
    for r0 in range(0, N, step):
        n = min(step, N - r0)
        out[r0:r0 + n, :C * F] = (q[r0:r0 + n, :, None] * h[r0:r0 + n, None, :]).reshape(n, C * F)
        out[r0:r0 + n, C * F:D] = q[r0:r0 + n]
    return out, y


def _rows(case, seed):
    g, dtype = _generator(seed), DTYPES[case["dtype"]]
    if case["rows"] == "lowrank":
        return _lowrank(g, case["N"], case["D"], dtype, case["aligned"])
    if case["rows"] == "lastlayer":
        return _lastlayer(g, case["N"], case["C"], case["D"], dtype, case["aligned"])[0]
    w = workloads.WORKLOADS["c4" if case["rows"] == "long" else "c5"]
    w = workloads.scaled(w, N=case["N"], D=case["D"], chunk_rows=case["N"])
    return workloads.DeviceStream(w, seed).chunk(0)


def prepare(case, seed):
    """Rows (or factors, or scores) on the device, and the handle that a program keeps from epoch to epoch."""
    kind = case["kind"]
    if kind == "select":
        return {"case": case, "scores": torch.tanh(0.5 * _rand(_generator(seed), case["N"]))}
    dtype = DTYPES[case["dtype"]]
    if kind == "host":
        return {"case": case, "rows": _rows(case, seed).cpu().pin_memory()}
    if kind == "factors":
        q, h, _ = _head(_generator(seed), case["N"], case["C"], case["F"])
        eb = 4 if dtype == torch.float32 else 2
        fac = []
        for t in (q, h):
            p = torch.zeros((t.shape[0], workloads.padded_pitch(t.shape[1], eb)), dtype=dtype, device="cuda")
            p[:, :t.shape[1]] = t
            fac.append(p)
        D = case["C"] * case["F"] + case["C"]
        return {"case": case, "q": fac[0], "h": fac[1], "fd": sage.SageFD(D, case["ell"], dtype, 0)}
    fd = sage.SageFD(case["D"], case["ell"], dtype, 0)
    if kind == "score":
        g = _generator(seed)
        rows, y = _lastlayer(g, case["N"], case["C"], case["D"], dtype, case["aligned"])
        # a sketch of the rows' own span with a decaying spectrum: random combinations of some of them
        some = rows[torch.randint(case["N"], (4 * case["ell"],), generator=g, device="cuda"), :case["D"]].float()
        S = _rand(g, case["ell"], some.shape[0]) @ some / math.sqrt(some.shape[0])
        S *= torch.linspace(1.0, 0.05, case["ell"], device="cuda")[:, None]
        fd.load_sketch(S)
        torch.cuda.synchronize()
        return {"case": case, "rows": rows, "labels": y, "fd": fd}
    if case["sketches"] > 1:
        fd.set_option(6, case["sketches"])
    return {"case": case, "rows": _rows(case, seed), "fd": fd}


# ---- one pass --------------------------------------------------------------------------------------------------

def _calls(n, chunk):
    step = chunk or n
    return [(r0, min(n, r0 + step)) for r0 in range(0, n, step)]


def _mask(scores, idx):
    return torch.zeros(scores.shape, dtype=torch.bool, device=scores.device).index_fill_(0, idx, True)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "select":
        return sage.sage_select(state["scores"], case["keep"])
    if kind == "host":
        return _host(state["rows"], case)
    fd = state["fd"]
    if kind == "score":
        fd.score(state["rows"])
        scores = fd.score_classes(state["labels"], case["C"])
        idx, per_class = sage.sage_select_classes(scores, state["labels"], case["C"], case["keep"])
        return {"scores": scores, "kept": _mask(scores, idx), "per_class": torch.tensor(per_class)}
    fd.reset()
    if kind == "factors":
        q, h, C, F = state["q"], state["h"], case["C"], case["F"]
        for a, b in _calls(case["N"], case["chunk"]):
            fd.update_outer(q[a:b], h[a:b], C, F)
        fd.finalize()
        scores = fd.score_outer(q, h, C, F)
    else:
        rows = state["rows"]
        for a, b in _calls(case["N"], case["chunk"]):
            fd.update(rows[a:b])
        fd.finalize()
        scores = fd.score(rows)
    _, sigma = fd.sketch()
    return {"sigma": sigma, "scores": scores, "kept": _mask(scores, sage.sage_select(scores, case["keep"]))}


def _host(rows, case):
    scores, idx = sage.sage_select_from_host(rows, case["D"], case["ell"], case["keep"], case["chunk"])
    return {"scores": scores, "kept": _mask(scores, idx)}


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def work(case):
    N, kind = case["N"], case["kind"]
    k = sage_count(N, case["keep"])
    if kind == "select":
        return {"bytes": 4 * N + 8 * k, "flops": 0}
    ell, m = case["ell"], 2 * case["ell"]
    eb = 4 if case["dtype"] == "f32" else 2
    D = case["C"] * case["F"] + case["C"] if kind == "factors" else case["D"]
    row_bytes = eb * (case["C"] + case["F"] if kind == "factors" else D)
    if kind == "score":
        return {"bytes": N * row_bytes + 4 * ell * D + 4 * N + 4 * N + N, "flops": 2 * N * ell * D + 4 * N * ell}
    # shrinks: one when the first 2 ell rows are in, then one every ell + 1 rows; each takes the inner products of its
    # new rows with the buffer, an m x m eigen-problem and the product that rebuilds ell - 1 rows
    shrinks = max(0, (N - m) // (ell + 1) + 1 if N >= m else 0) + 1
    project = 2 * N * ell * (case["C"] * (case["F"] + 2) if kind == "factors" else D)
    kept = 0 if kind == "host" else 4 * ell * D + 4 * ell
    return {"bytes": N * row_bytes + kept + 4 * N + N, "flops": shrinks * (2 * (ell + 1) * m * D + 9 * m ** 3 + 2 * (ell - 1) * m * D) + project}


def sage_count(N, keep):
    return max(0, min(N, int(math.floor(keep * N + 0.5))))


def tolerance(case):
    """Four times the largest difference from an fp64 replay of the path (scores and row norms; f32 rows and bf16 rows
    of less than 16,384 values: 1e-5 and 3.2e-7 more for every shrink, as the fp32 Gram matrices of a long chain all
    round the same way; longer bf16 rows meet a bf16 sketch: 1.8e-3, single scores 6.2e-3). One kept example in 10,000 was
    another one than in fp64; at least one pair may trade places."""
    if case["kind"] == "select":
        return "exact"
    N, ell = case["N"], case["ell"]
    D = case["C"] * case["F"] + case["C"] if case["kind"] == "factors" else case["D"]
    shrinks = 0 if case["kind"] == "score" else N / (ell + 1) / case.get("sketches", 1)
    rel = 4 * (1e-5 + 3.2e-7 * shrinks)
    differ = max(4e-4, 2.0 / N)
    if case["dtype"] == "bf16" and D >= 16384:
        return {"rel": 7e-3, "max": 2.5e-2, "differ": differ}
    return {"rel": rel, "max": 4 * rel, "differ": differ}
