"""Timed cases of the simulator: whole runs, the block codec, the size predictor's training and the readout.

Each case goes through the package's public calls the way a user's program does: a plan is made once and run, a block
is compressed or decompressed, the predictor is trained on logged rows, amplitudes of a finished state are read.
`listed()` gives the fixed cases, `draw(rng)` more of the same ranges. `exact()` gives a case's outputs in 64 bits
from plain torch: the full state vector of a circuit gate by gate, or the codec's rounding of a block.
"""
import math

import numpy as np
import torch

from paper_2410_14088_gb300 import inputs, qsim

TCGEN05 = {"prec": "tf32", "k": 5, "tcgen05": 1, "reorder": 2, "diag_exempt": 1}


def listed():
    return [
        # The smallest whole run: 16 qubits, 64 blocks of 2^10 amplitudes, plain FP32 gates. A parameter study runs
        # thousands of these; launches and the calls around them count.
        dict(_run("random", 16, 8, 10, 2), name="run_random16_fp32", k=4),
        # QFT of a basis state, then RZ and CX layers, on 28 qubits with 2^22-amplitude blocks; gates fused to five
        # qubits in TF32 on the tensor cores.
        dict(_run("qft", 28, 4, 22, 4), name="run_qft28_tf32", **TCGEN05),
        # QAOA MaxCut, three layers, in the form of the default benchmark (TF32 on the tensor cores, learned sizing,
        # blocks of 2^25, inner size 3) on 30 qubits, the largest state read back whole here.
        dict(_run("qaoa", 30, 3, 25, 3), name="run_qaoa30_tf32_learned", sizing="predict", **TCGEN05),
        # Random brick circuit of depth 14 with plain FP32 gates: every value within 1e-5 of 64 bits before the codec.
        dict(_run("random", 26, 14, 22, 4), name="run_random26_fp32", k=4, reorder=2, diag_exempt=1),
        # The relative-bound codec with split-BF16 gates (FP32-like accuracy on the tensor cores), an odd qubit count.
        dict(_run("random", 25, 8, 20, 3), name="run_random25_bf16x3_rel", codec="rel", prec="bf16x3", k=5, tcgen05=1,
             reorder=2, diag_exempt=1),
        # Sixteen independent circuits of uneven size (GHZ, QFT, random, Grover; 17 to 22 qubits) in one persistent
        # launch with learned sizing: a service working off a queue of jobs.
        {"name": "batch16_persistent", "kind": "batch", "count": 16, "nmin": 17, "nmax": 22, "inner": 2, "eps": 1e-3},
        # One small block compressed: the smallest codec call, where latency counts.
        _block("compress", 10, "gaussian", "abs", "compress_m10"),
        # One block of 2^22 amplitudes with the statistics of a random state, the benchmark's middle block size.
        _block("compress", 22, "gaussian", "abs", "compress_m22"),
        # The same block back again: what every stage does to every block it reads.
        _block("decompress", 22, "gaussian", "abs", "decompress_m22"),
        # The relative bound (sign and logarithm) on a block with a slowly varying phase, as after a QFT.
        _block("compress", 20, "smooth", "rel", "compress_rel_m20"),
        # The size predictor trained on the rows two logged runs give, with the benchmark's settings.
        {"name": "train_1280", "kind": "train", "rows": 1280, "epochs": 40, "batch": 64},
        # Sampled amplitudes of a finished 26-qubit state: what a user reads from a state too large to print.
        dict(_run("random", 26, 4, 20, 3), name="amplitudes_65536", kind="amplitudes", count=65536, k=4),
    ]


def draw(rng):
    kind = rng.choice(["run"] * 5 + ["compress"] * 2 + ["decompress"] * 2 + ["batch", "train", "amplitudes"])
    if kind in ("compress", "decompress"):
        return _block(kind, rng.randint(5, 24), rng.choice(["gaussian", "smooth", "sparse"]), rng.choice(["abs", "abs", "rel"]),
                      n_equiv=rng.randint(10, 32))
    if kind == "train":
        return {"kind": kind, "rows": _log(rng, 64, 4000), "epochs": rng.randint(1, 20), "batch": rng.choice([16, 64, 100, 256])}
    if kind == "batch":
        nmin = rng.randint(16, 18)
        return {"kind": kind, "count": rng.randint(2, 20), "nmin": nmin, "nmax": rng.randint(nmin, 21),
                "inner": rng.randint(2, 4), "eps": rng.choice([1e-2, 1e-3])}
    n = rng.randint(12, 26)
    circuit = rng.choice(["random", "random", "qft", "qaoa", "ghz", "grover"])
    if circuit == "qaoa":
        n -= n % 2  # a 3-regular graph has an even number of vertices
    size = {"random": rng.randint(2, 14), "qft": rng.randint(0, 4), "qaoa": rng.randint(1, 3), "ghz": 0, "grover": rng.randint(3, 6)}[circuit]
    inner = rng.randint(2, 4)
    m = rng.randint(max(5, n - 10), n - inner)
    c = _run(circuit, n, size, m, inner, eps=rng.choice([1e-2, 1e-3]))
    c["prec"] = rng.choice(["fp32", "tf32", "tf32", "bf16x3"])
    c["k"] = rng.randint(2, 5)
    c["tcgen05"] = rng.choice([0, 1]) if c["prec"] != "fp32" else 0
    c["reorder"] = rng.choice([0, 2])
    c["diag_exempt"] = rng.choice([0, 1])
    c["codec"] = rng.choice(["abs", "abs", "abs", "rel", "none"])
    if c["codec"] != "none":
        c["sizing"] = rng.choice(["exact", "exact", "predict"])
        c["mode"] = rng.choice(["streams", "streams", "persistent"]) if m >= 12 else "streams"
    c["streams"] = rng.choice([1, 2, 4])
    c["kind"] = kind
    if kind == "amplitudes":
        c["count"] = _log(rng, 1, 200000)
    return c


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("run", "amplitudes"):
        if case.get("sizing") == "predict":
            _trained_predictor()
        plan = qsim.plan_stages(_circuit(case, seed), **_options(case))
        if kind == "run":
            return {"kind": kind, "plan": plan}
        return {"kind": kind, "state": qsim.run(plan), "idx": _indices(case, seed)}
    if kind == "batch":
        _trained_predictor()
        plans = []
        for c in _batch(case, seed):
            plans.append(qsim.plan_stages(c, m=max(5, min(26, c.n - 4)), inner=case["inner"], k=5, prec=qsim.PREC_TF32, tcgen05=1,
                                          mode=qsim.MODE_PERSISTENT, sizing=qsim.SIZING_PREDICT, predictor_margin=0.25,
                                          reorder=2, diag_exempt=1, eps=case["eps"]))
        return {"kind": kind, "plans": plans}
    if kind == "train":
        return {"kind": kind, "rows": _rows(case, seed).cpu().numpy(), "epochs": case["epochs"], "batch": case["batch"]}
    x = _amps(case, seed)
    m, rel = case["m"], case["codec"] == "rel"
    if kind == "compress":
        out = torch.zeros((qsim.qszr_worst_case_bytes if rel else qsim.worst_case_bytes)(m), dtype=torch.uint8, device="cuda")
        return {"kind": kind, "x": x, "m": m, "rel": rel, "bound": _bound(case), "out": out}
    out, nb = (qsim.compress_block_rel if rel else qsim.compress_block)(x, m, _bound(case))
    return {"kind": kind, "stream": out[:nb].clone(), "m": m}


def run(state):
    kind = state["kind"]
    if kind == "run":
        return qsim.run(state["plan"]).decompress()
    if kind == "batch":
        states, _ = qsim.run_batch(state["plans"])
        return [s.decompress() for s in states]
    if kind == "compress":
        compress = qsim.compress_block_rel if state["rel"] else qsim.compress_block
        out, nb = compress(state["x"], state["m"], state["bound"], out=state["out"])
        return {"stream": out, "bytes": nb}
    if kind == "decompress":
        return qsim.decompress_block(state["stream"], state["m"])
    if kind == "train":
        loss = qsim.predictor_train(state["rows"], epochs=state["epochs"], batch=state["batch"], lr=3e-3, seed=100)
        return {"loss": loss, "params": qsim.predictor_get()}
    return state["state"].amplitudes(state["idx"])


def work(case):
    kind = case["kind"]
    if kind == "run":  # nothing to read but the gates; every gate's update, and the state written once
        gates = _circuit(case, 1).gates
        return {"bytes": 8.0 * 2 ** case["n"], "flops": 2.0 ** case["n"] * sum(map(_gate_flops, gates))}
    if kind == "batch":
        cs = _batch(case, 1)
        return {"bytes": sum(8.0 * 2 ** c.n for c in cs), "flops": sum(2.0 ** c.n * sum(map(_gate_flops, c.gates)) for c in cs)}
    if kind == "train":  # two flops per weight forward, four backward, ten per weight for Adam's step
        rows, steps = case["rows"] * case["epochs"], case["epochs"] * -(-case["rows"] // case["batch"])
        return {"bytes": 4.0 * (case["rows"] * qsim.TRAIN_ROW + qsim.MLP_PARAMS),
                "flops": float(qsim.MLP_PARAMS) * (6 * (rows + case["rows"]) + 10 * steps)}
    if kind == "amplitudes":  # the indices in, the amplitudes out, and the compressed values they come from
        return {"bytes": (8.0 + 8.0 + 3.0) * case["count"], "flops": 0.0}
    ratio = {"gaussian": 2.8, "smooth": 4.0, "sparse": 20.0}[case["block"]] / (1.7 if case["codec"] == "rel" else 1.0)
    return {"bytes": 8.0 * 2 ** case["m"] * (1 + 1 / ratio), "flops": 0.0}


def exact(case, seed):
    kind = case["kind"]
    if kind == "run":
        return _ideal(_circuit(case, seed))
    if kind == "batch":
        return [_ideal(c) for c in _batch(case, seed)]
    if kind == "amplitudes":
        psi = _ideal(_circuit(case, seed))
        return psi[torch.from_numpy(_indices(case, seed).astype(np.int64)).cuda()]
    if kind == "train":
        return _train64(case, seed)
    if kind == "compress":
        return None  # bytes: equal or not
    x = torch.view_as_real(_amps(case, seed))
    if case["codec"] == "rel":
        k = max(k for k in range(1, 23) if 2.0 ** (k - 24) <= case["rel"] / (1 + case["rel"]))
        u = x.contiguous().view(torch.int32) & 0x7FFFFFFF
        mag = (((u + (1 << (k - 1))) >> k) << k).view(torch.float32).double()
        y = torch.where(x < 0, -mag, mag)
    else:
        step = 2.0 ** (math.frexp(2 * _bound(case))[1] - 1)
        y = torch.round(x.double() / step) * step
    return torch.view_as_complex(y.contiguous())


# ---- the cases' descriptions ---------------------------------------------------------------------------------------

def _run(circuit, n, size, m, inner, eps=1e-3):
    return {"kind": "run", "circuit": circuit, "n": n, "size": size, "m": m, "inner": inner, "eps": eps}


def _block(kind, m, block, codec, name=None, n_equiv=None):
    c = {"kind": kind, "m": m, "block": block, "codec": codec, "rel": 1e-3, "n_equiv": n_equiv or m + 6}
    return dict(c, name=name) if name else c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _options(case):
    kw = {f: case[f] for f in ("m", "inner", "eps", "k", "tcgen05", "reorder", "diag_exempt", "streams") if f in case}
    kw["prec"] = {"fp32": qsim.PREC_FP32, "tf32": qsim.PREC_TF32, "bf16x3": qsim.PREC_BF16X3}[case.get("prec", "fp32")]
    kw["codec"] = {"abs": qsim.CODEC_QSZ1, "rel": qsim.CODEC_QSZR, "none": qsim.CODEC_NONE}[case.get("codec", "abs")]
    if case.get("sizing") == "predict":
        kw.update(sizing=qsim.SIZING_PREDICT, predictor_margin=0.25)
    if case.get("mode") == "persistent":
        kw.update(mode=qsim.MODE_PERSISTENT, graph=1)
    return kw


# ---- inputs --------------------------------------------------------------------------------------------------------

def _circuit(case, seed):
    n, size = case["n"], case["size"]
    if case["circuit"] == "random":
        return inputs.random_brick(n, size, seed)
    if case["circuit"] == "qft":
        return inputs.qft_rz_cx(n, size, seed)
    if case["circuit"] == "qaoa":
        return inputs.qaoa_maxcut(n, size, seed)
    basis = inputs.SplitMix64(seed).next_u64() >> (64 - n)
    if case["circuit"] == "grover":
        return inputs.grover(n, size, basis)
    c = inputs.ghz(n)
    c.init_basis = basis
    return c


def _batch(case, seed):
    sub, span, cs = inputs.SplitMix64(seed), case["nmax"] - case["nmin"] + 1, []
    for i in range(case["count"]):
        circuit = ("ghz", "qft", "random", "grover")[i % 4]
        size = {"ghz": 0, "qft": 0, "random": 8, "grover": 3 + i // 4 % 4}[circuit]
        cs.append(_circuit({"circuit": circuit, "n": case["nmin"] + 5 * i % span, "size": size}, sub.next_u64()))
    return cs


def _indices(case, seed):
    return np.random.default_rng(seed).integers(0, 1 << case["n"], case["count"], dtype=np.uint64)


def _bound(case):
    return case["rel"] if case["codec"] == "rel" else 1e-3 * 2.0 ** (-case["n_equiv"] / 2)


def _amps(case, seed):
    """2^m complex64 amplitudes of a block of an n_equiv-qubit state."""
    N, g = 1 << case["m"], torch.Generator(device="cuda").manual_seed(seed)
    size = 2.0 ** (-case["n_equiv"] / 2)
    if case["block"] == "gaussian":  # a random state's amplitudes
        return torch.view_as_complex(torch.randn(N, 2, generator=g, device="cuda") * (size * math.sqrt(0.5)))
    if case["block"] == "smooth":  # flat magnitude, slowly varying phase
        u = torch.rand(2, generator=g, device="cuda", dtype=torch.float64)
        phase = 2 * math.pi * (u[0] + u[1] * torch.arange(N, device="cuda", dtype=torch.float64) / N * 7.0)
        return torch.polar(torch.full_like(phase, size), phase).to(torch.complex64)
    x = torch.zeros(N, 2, device="cuda")  # a few large amplitudes
    at = torch.randperm(N, generator=g, device="cuda")[:max(1, N // 4096)]
    x[at] = torch.rand(at.numel(), 2, generator=g, device="cuda") - 0.5
    return torch.view_as_complex(x)


def _trained_predictor():
    """The predictor's weights from the rows of one logged run, as a program sets them up before learned sizing."""
    c = inputs.random_brick(16, 4, 5)
    rows = qsim.run(qsim.plan_stages(c, m=10, inner=2, k=4, collect=1)).training_data()
    qsim.predictor_train(rows, epochs=4, batch=64, lr=3e-3, seed=100)


def _rows(case, seed):
    """Training rows as runs log them: a block's histogram of code lengths (a peak of some width), its largest bin, the
    stage's features, and the log2 of its compressed share."""
    g, n = torch.Generator(device="cuda").manual_seed(seed), case["rows"]

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(n, *shape, generator=g, device="cuda")

    centre, width, zeros = uniform(2, 14, 1), uniform(0.4, 1.5, 1), uniform(0, 0.5, 1)
    bins = torch.arange(32, device="cuda")
    hist = torch.exp(-((bins - centre) / width) ** 2)
    hist = hist / hist.sum(1, keepdim=True) * (1 - zeros)
    hist[:, :1] += zeros
    top = (bins * (hist > 1e-4)).amax(1, keepdim=True) / 32
    target = torch.log2(((1 - zeros) * (centre + 1.5) + 0.3) / 32) + 0.05 * torch.randn(n, 1, generator=g, device="cuda")
    return torch.cat([hist, top, uniform(0, 1, 8), target], 1)


# ---- 64-bit references ---------------------------------------------------------------------------------------------

def _gate_flops(g):
    """Flops per amplitude of the state: a dense one-qubit update 14, a phase 6 on the amplitudes that it changes."""
    if g.phaseflip or g.name == "cx":
        return 0.0
    if g.is_diagonal:
        return 6.0 * float(np.mean(np.diag(g.matrix) != 1))
    return 14.0


def _ideal(c):
    psi = torch.zeros(1 << c.n, dtype=torch.complex128, device="cuda")
    psi[c.init_basis] = 1
    for g in c.gates:
        if g.phaseflip:
            psi[g.basis] *= -1
            continue
        order = sorted(g.qubits)
        v = psi.view([-1, 2, 1 << order[0]] if len(order) == 1 else [-1, 2, 1 << (order[1] - order[0] - 1), 2, 1 << order[0]])
        parts = []
        for r in range(1 << len(order)):  # the slice whose qubits spell matrix row r
            bit = {q: (r >> j) & 1 for j, q in enumerate(g.qubits)}
            parts.append(v[:, bit[order[0]]] if len(order) == 1 else v[:, bit[order[1]], :, bit[order[0]]])
        if g.is_diagonal:
            for r, p in enumerate(parts):
                if g.matrix[r, r] != 1:
                    p *= complex(g.matrix[r, r])
            continue
        changed = [r for r in range(len(parts)) if np.any(g.matrix[r] != np.eye(len(parts))[r])]
        old = {r: parts[r].clone() for r in changed}
        for r in changed:
            parts[r].zero_()
            for s in range(len(parts)):
                if g.matrix[r, s] != 0:
                    parts[r].add_(old.get(s, parts[s]), alpha=complex(g.matrix[r, s]))
    return psi


def _train64(case, seed):
    """He-uniform weights from splitmix64, Fisher-Yates order from the same stream, Adam on 0.5 (y - t)^2, in 64 bits."""
    data = _rows(case, seed).double()
    x, t = data[:, :41], data[:, 41]
    rng, p = inputs.SplitMix64(100), []
    for out, fan in ((64, 41), (64, 64), (1, 64)):
        u = np.array([rng.uniform() for _ in range(out * fan)])
        w = ((2 * u - 1) * math.sqrt(6.0 / fan)).astype(np.float32).reshape(out, fan)
        p += [torch.from_numpy(w).cuda().double(), torch.zeros(out, dtype=torch.float64, device="cuda")]

    def step(rows):
        a1 = x[rows] @ p[0].T + p[1]
        h1 = a1.relu()
        a2 = h1 @ p[2].T + p[3]
        h2 = a2.relu()
        r = (h2 @ p[4].T + p[5]).squeeze(1) - t[rows]
        dy = (r / r.numel())[:, None]
        d2 = dy @ p[4] * (a2 > 0)
        d1 = d2 @ p[2] * (a1 > 0)
        return 0.5 * (r * r).mean(), [d1.T @ x[rows], d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0)]

    lr, b1, b2, eps = (float(np.float32(v)) for v in (3e-3, 0.9, 0.999, 1e-8))
    first, second, n = [torch.zeros_like(w) for w in p], [torch.zeros_like(w) for w in p], 0
    for _ in range(case["epochs"]):
        perm = list(range(case["rows"]))
        for i in range(case["rows"] - 1, 0, -1):
            j = rng.next_u64() % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        perm = torch.tensor(perm, device="cuda")
        for at in range(0, case["rows"], case["batch"]):
            n += 1
            for w, g, a, b in zip(p, step(perm[at:at + case["batch"]])[1], first, second):
                a.mul_(b1).add_(g, alpha=1 - b1)
                b.mul_(b2).addcmul_(g, g, value=1 - b2)
                w -= lr * (a / (1 - b1 ** n)) / ((b / (1 - b2 ** n)).sqrt() + eps)
    return {"loss": step(slice(None))[0], "params": torch.cat([w.reshape(-1) for w in p])}
