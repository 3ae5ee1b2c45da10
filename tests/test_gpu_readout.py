"""Readout of finished states: what the calls leave behind on an error."""
import ctypes

import numpy as np
import pytest

from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("codec", [qsim.CODEC_QSZ1, qsim.CODEC_QSZR])
def test_amplitudes_written_whole_or_not_at_all(codec):
    """A request longer than the library takes at a time (2^24 indices) whose last index is in a block that cannot be
    read: one rank's state of a sharded run, where the other rank's blocks are missing."""
    c = inputs.Circuit(16, [inputs.H(0), inputs.H(9), inputs.CZ(9, 10)])
    plan = qsim.plan_stages(c, m=9, inner=2, k=4, eps=1e-3, codec=codec)
    run = qsim.ShardRun(plan, plan.shards(1), 1, 1)
    for s in range(plan.nstages):
        run.stage(s)
    st = run.finish()
    held = [b for b in range(1 << 7) if st.block_stream(b)]
    assert held and len(held) < 1 << 7
    missing = next(b for b in range(1 << 7) if b not in held)
    for count in (5, (1 << 24) + 3):
        idx = np.full(count, held[0] << 9, dtype=np.uint64)
        out = np.full(2 * count, 7.0, dtype=np.float32)
        call = lambda: qsim.lib().qsim_amplitudes(st.handle, idx.ctypes.data_as(ctypes.POINTER(ctypes.c_uint64)), count,
                                                  out.ctypes.data_as(ctypes.POINTER(ctypes.c_float)))
        idx[-1] = (missing << 9) + 3
        assert call() == qsim.E_CORRUPT
        assert (out == 7.0).all()
        idx[-1] = (held[-1] << 9) + 3
        assert call() == qsim.OK
        want = st.amplitudes(idx[-2:])
        assert (out.view(np.complex64)[:-1] == want[0]).all() and out.view(np.complex64)[-1] == want[1]


def test_decompressing_an_uncompressed_state_takes_little_scratch():
    c = inputs.random_brick(24, 1, 3)
    st = qsim.run(qsim.plan_stages(c, m=5, inner=2, k=2, codec=qsim.CODEC_NONE))  # 2^19 blocks
    small = qsim.run(qsim.plan_stages(inputs.random_brick(10, 1, 3), m=5, inner=2, k=2, codec=qsim.CODEC_NONE))
    small.decompress()  # the kernels are loaded
    out = torch.empty(1 << 24, dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    qsim.release_cached_memory()
    free, _ = torch.cuda.mem_get_info()
    st.decompress(out=out)
    assert free - torch.cuda.mem_get_info()[0] <= 4 << 20  # 2^16 references of 16 bytes, in cudaMalloc's units of 2 MB
    idx = np.array([0, 31, 32, (1 << 21) - 1, 1 << 21, (1 << 24) - 1], dtype=np.uint64)  # across the lists' ends
    np.testing.assert_array_equal(out.cpu().numpy()[idx.astype(np.int64)], st.amplitudes(idx))
