"""The persistent kernel's size prediction sums the output layer with fused products, as qsim_mlp_forward does."""
import numpy as np
import pytest

from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_output_layer_is_fused():
    # one live unit per layer: h1[0] = 1, h2[0] = 5001, y = 5001 h2[0] + b3. 5001^2 = 25010001 is odd above 2^24, so a
    # product rounded to FP32 is 25010000 and y loses 1: every block's slot halves
    p = np.zeros(qsim.MLP_PARAMS, dtype=np.float32)
    ob1, ow2 = 64 * 41, 64 * 41 + 64
    ow3 = ow2 + 64 * 64 + 64
    p[ob1], p[ow2], p[ow3], p[ow3 + 64] = 1.0, 5001.0, 5001.0, -25010004.0
    qsim.predictor_set(p)
    y = qsim.mlp_forward(torch.from_numpy(p).cuda(), torch.zeros(1, 41, device="cuda"))
    assert y.item() == -3.0
    c = inputs.ghz(14)
    st = qsim.run(qsim.plan_stages(c, m=10, inner=2, k=2, mode=qsim.MODE_PERSISTENT, sizing=qsim.SIZING_PREDICT,
                                   predictor_margin=0.0))
    assert st.stats.overflow_blocks == 0
    assert st.stats.peak_reserved_bytes == (1 << 4) * (1 << (10 + 3 - 3))  # 2^(m + 3 + y) bytes per block
