"""Tile passes that keep their tiles in registers (stream engine) against the staged form of the same passes, which the
persistent kernel runs: the operands, their order and every rounding are the same, so the stored streams are equal
bytes. Circuits with one to many width-5 dense ops per pass (B operands kept, or reloaded per op), ops on the tile's
lowest bits at either end (groups through the staged tile) and away from them (straight from and to memory), runs of
diagonal ops before, between and after the dense ops, a single tile, and odd numbers of tiles."""
import numpy as np
import pytest

import oracle
from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def layered(n, qubits, layers, seed, diag):
    """Layers of U3 on the given qubits, CZ chains on them between layers so that they fuse to wide ops, and diagonal
    layers (RZZ over all qubits, RZ) where diag has the layer."""
    rng, gates = inputs.SplitMix64(seed), []
    for layer in range(layers):
        if layer in diag:
            for q in range(n):
                gates.append(inputs.RZZ(q, (q + 1 + layer) % n, 3.0 * rng.uniform()))
                gates.append(inputs.RZ(q, 3.0 * rng.uniform()))
        for q in qubits[layer % len(qubits)]:
            gates.append(inputs.U3(q, *(6.28 * rng.uniform() for _ in range(3))))
        ring = qubits[layer % len(qubits)]
        for a, b in zip(ring, ring[1:]):
            gates += [inputs.CX(a, b), inputs.U3(b, *(6.28 * rng.uniform() for _ in range(3)))]
    return inputs.Circuit(n, gates, 0)


LOW, MID, HIGH = (0, 1, 2, 3, 4), (5, 6, 7, 8, 9), (7, 8, 9, 10, 11)
CASES = [
    (12, [MID], 1, (), 12, 2),            # one tile, one op, groups straight from and to memory
    (13, [LOW], 1, (), 13, 2),            # two tiles, the op on the lowest bits
    (15, [MID, LOW], 2, (), 13, 2),       # in straight, out staged
    (15, [LOW, MID], 2, (1,), 13, 2),     # in staged, a run between
    (16, [MID, HIGH], 4, (0, 2), 14, 2),  # runs first and between
    (16, [HIGH, MID, LOW], 9, (3, 9), 14, 2),
    (17, [HIGH, (3, 5, 7, 9, 11), (3, 4, 6, 8, 10)], 6, (0, 1, 2, 3, 4, 5), 13, 3),
]


@pytest.mark.parametrize("prec", [qsim.PREC_TF32, qsim.PREC_BF16X3], ids=["tf32", "bf16x3"])
@pytest.mark.parametrize("n,qubits,layers,diag,m,inner", CASES)
def test_same_bytes_as_the_staged_form(n, qubits, layers, diag, m, inner, prec):
    c = layered(n, qubits, layers, 31 + n, diag)
    kw = dict(m=min(m, n), inner=inner, k=5, prec=prec, tcgen05=1, reorder=2, diag_exempt=1)
    a = qsim.run(qsim.plan_stages(c, streams=2, **kw))
    b = qsim.run(qsim.plan_stages(c, mode=qsim.MODE_PERSISTENT, graph=1, **kw))
    for blk in range(1 << (n - kw["m"])):
        assert a.block_stream(blk) == b.block_stream(blk)
    raw = qsim.run(qsim.plan_stages(c, codec=qsim.CODEC_NONE, **kw)).decompress().cpu().numpy()
    plan = qsim.plan_stages(c, codec=qsim.CODEC_NONE, **kw)
    ops = sum(1 for s in range(plan.nstages) for o in plan.stage_ops(s) if o["type"] == 0)
    # TF32 rounds both operands of an op to 2^-11: at most 2^-10 of the norm per op; split BF16: below 2^-20
    want = oracle.simulate(c)
    assert np.linalg.norm(raw - want) <= ops * (2.0 ** -10 if prec == qsim.PREC_TF32 else 2.0 ** -20)
