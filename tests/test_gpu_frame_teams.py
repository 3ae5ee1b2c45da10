"""The frame coder with one thread per chunk pair, at the edges of its shapes: every frame size (1 to 128 chunks per
plane, one to four warps), codes of up to 16 bits and wider (the two register transposes), all-zero frames between
others, and an output that is only 8-byte aligned. Streams and decoded values are compared with the scalar oracle
exactly: they are integers scaled by a power of two, so the tolerance is zero."""
import numpy as np
import pytest

import oracle
from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def block(m, wide, seed):
    """Gaussian amplitudes, frames 1, 4, 7, ... all zero; wide: codes of up to 27 bits in every other chunk."""
    x = inputs.gaussian_block(m, 14, seed).reshape(-1, 2)
    if wide:
        x[32::64] *= 2.0 ** 12
        x[5] *= 2.0 ** 14
    F = min(1 << m, 4096)
    for f in range(1, len(x) // F, 3):
        x[f * F:(f + 1) * F] = 0
    return np.ascontiguousarray(x.reshape(-1))


@pytest.mark.parametrize("codec", ["abs", "rel"])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("m", [5, 6, 7, 8, 9, 10, 11, 12, 13, 15])
def test_decode_matches_oracle(m, wide, codec):
    x = block(m, wide, 77 + m)
    eb = 1e-3 * 2.0 ** -7
    stream = oracle.qsz_encode(x, m, eb) if codec == "abs" else oracle.qszr_encode(x, m, 1e-3)
    want = oracle.qsz_decode(stream, m) if codec == "abs" else oracle.qszr_decode(stream, m)
    buf = torch.frombuffer(bytearray(stream), dtype=torch.uint8).cuda()
    got = qsim.decompress_block(buf, m).cpu().numpy().view(np.float32)
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("codec", ["abs", "rel"])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("m", [5, 6, 7, 8, 9, 10, 11, 12, 13, 15])
def test_encode_matches_oracle(m, wide, codec):
    x = block(m, wide, 177 + m)
    eb = 1e-3 * 2.0 ** -7
    dev = torch.from_numpy(x).cuda()
    if codec == "abs":
        out, nb = qsim.compress_block(dev, m, eb)
        want = oracle.qsz_encode(x, m, eb)
    else:
        out, nb = qsim.compress_block_rel(dev, m, 1e-3)
        want = oracle.qszr_encode(x, m, 1e-3)
    assert out[:nb].cpu().numpy().tobytes() == want
    np.testing.assert_array_equal(dev.cpu().numpy(), x)  # the input is not modified


@pytest.mark.parametrize("value", [16383.0, 16383.5, 16384.0, 2.0 ** 22, 2.0 ** 29])
def test_codes_at_the_edge_of_the_packed_form(value):
    """Codes of both signs around +-16383 steps, the largest the packed 16-bit differences hold, and far beyond."""
    m, eb = 6, 0.5  # step 1
    x = np.zeros((64, 2), dtype=np.float32)
    x[7], x[8], x[40, 1] = value, -value, -value
    x = x.reshape(-1)
    out, nb = qsim.compress_block(torch.from_numpy(x).cuda(), m, eb)
    assert out[:nb].cpu().numpy().tobytes() == oracle.qsz_encode(x, m, eb)


@pytest.mark.parametrize("codec", [qsim.CODEC_QSZ1, qsim.CODEC_QSZR])
@pytest.mark.parametrize("m", [9, 12, 13, 15])
def test_stored_streams_are_the_oracles(m, codec):
    """Blocks of one frame go straight to their slots, larger ones through the copy: the stored stream of every block
    equals the oracle's stream of the block's values, and two runs store the same bytes."""
    c = inputs.random_brick(17, 3, 8)
    plan = qsim.plan_stages(c, m=m, inner=2, k=4, codec=codec)
    st, again = qsim.run(plan), qsim.run(plan)
    amps = st.decompress().cpu().numpy().view(np.float32).reshape(-1, 2 << m)
    for b in range(1 << (17 - m)):
        got = st.block_stream(b)
        want = (oracle.qsz_encode(amps[b], m, 1e-3 * 2.0 ** -8.5) if codec == qsim.CODEC_QSZ1
                else oracle.qszr_encode(amps[b], m, 1e-3))
        assert got == want
        assert again.block_stream(b) == got


@pytest.mark.parametrize("codec", [qsim.CODEC_QSZ1, qsim.CODEC_QSZR])
def test_state_decompress_into_an_8_byte_aligned_tensor(codec):
    c = inputs.random_brick(15, 3, 4)
    st = qsim.run(qsim.plan_stages(c, m=13, inner=2, k=4, codec=codec))
    want = st.decompress()
    room = torch.zeros((1 << 15) + 1, dtype=torch.complex64, device="cuda")
    st.decompress(out=room[1:])
    assert torch.equal(room[1:], want)


@pytest.mark.parametrize("codec", [qsim.CODEC_QSZ1, qsim.CODEC_QSZR, qsim.CODEC_NONE])
@pytest.mark.parametrize("m", [5, 6, 7, 8, 10, 12, 14])
def test_single_amplitudes_equal_the_decompressed_state(m, codec):
    """Every index of a small state, unsorted and repeated, decoded one by one from its chunks."""
    c = inputs.random_brick(15, 4, 21)
    c.gates += [inputs.X(3), inputs.CP(2, 9, 0.3)]
    st = qsim.run(qsim.plan_stages(c, m=m, inner=2, k=4, codec=codec))
    idx = np.concatenate([np.random.default_rng(m).permutation(1 << 15), [0, 0, (1 << 15) - 1]]).astype(np.uint64)
    np.testing.assert_array_equal(st.amplitudes(idx), st.decompress().cpu().numpy()[idx.astype(np.int64)])
