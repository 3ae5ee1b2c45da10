"""Scratch of the persistent kernel: blocks of one frame keep no frame records."""
import pytest

from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_one_frame_blocks_keep_no_frame_records():
    kw = dict(m=5, inner=2, k=2, codec=qsim.CODEC_QSZR, eps=1e-3, mode=qsim.MODE_PERSISTENT)
    qsim.run(qsim.plan_stages(inputs.ghz(8), **kw))  # the kernels are loaded
    n, nblocks = 22, 1 << 17
    plan = qsim.plan_stages(inputs.Circuit(n, [inputs.H(0), inputs.CX(0, 6)]), **kw)
    qsim.release_cached_memory()
    free, _ = torch.cuda.mem_get_info()
    st = qsim.run(plan)
    used = free - torch.cuda.mem_get_info()[0]  # the state's, and what the library caches for the next run
    slot = -(-qsim.qszr_worst_case_bytes(5) // 256) * 256
    # the working vector, two arenas of worst-case slots, 64 MB for tables and descriptors; a record of 2048 bytes for
    # every block's frame would add 256 MB
    assert used <= (8 << n) + 2 * nblocks * slot + (64 << 20)
    assert abs(st.norm_sq() - 1) < 1e-2
