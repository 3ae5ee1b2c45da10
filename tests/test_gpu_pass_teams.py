"""Tile passes whose CTAs hold several tiles beside one pass blob: tiles of 2^8, 2^12 and 2^13 amplitudes (the last leave
room for fewer teams), fewer tiles than teams and many more, dense ops of every width on CUDA cores (several index groups
per thread at a time in 4096-amplitude tiles), against the FP64 oracle within the FP32 paths' 1e-5 per amplitude."""
import numpy as np
import pytest

import oracle
from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_bits", [8, 12, 13])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n,m", [(13, 11), (18, 14)])
def test_fp32_passes_match_fp64(n, m, k, tile_bits):
    c = inputs.random_brick(n, 5, 60 + k)
    if k == 1:  # single-qubit gates only
        c.gates = [g for g in c.gates if g.nq == 1]
    plan = qsim.plan_stages(c, m=m, inner=2, k=k, tile_bits=tile_bits, codec=qsim.CODEC_NONE)
    got = qsim.run(plan).decompress().cpu().numpy()
    assert np.max(np.abs(got - oracle.simulate(c))) <= 1e-5


@pytest.mark.parametrize("prec", [qsim.PREC_TF32, qsim.PREC_BF16X3], ids=["tf32", "bf16x3"])
@pytest.mark.parametrize("k", [3, 4, 5])
def test_warp_mma_passes_match_fp64(k, prec):
    c = inputs.random_brick(17, 6, 80 + k)
    plan = qsim.plan_stages(c, m=13, inner=2, k=k, prec=prec, codec=qsim.CODEC_NONE)
    got = qsim.run(plan).decompress().cpu().numpy()
    ops = sum(1 for s in range(plan.nstages) for o in plan.stage_ops(s) if o["type"] == 0)
    # both operands of an op rounded to TF32: at most 2^-10 of the norm per op; split BF16: below 2^-20
    assert np.linalg.norm(got - oracle.simulate(c)) <= ops * (2.0 ** -10 if prec == qsim.PREC_TF32 else 2.0 ** -20)
