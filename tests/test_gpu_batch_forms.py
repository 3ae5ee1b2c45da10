"""Batches whose plans differ in tcgen05: the tcgen05 form of the persistent kernel holds no warp-level MMAs, so circuits
that need them run in a launch of their own, and every circuit's streams equal those of the same plan run alone."""
import pytest

import oracle
from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu


def streams_of(st):
    return [st.block_stream(b) for b in range(1 << (st.n - st.m))]


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("prec", [qsim.PREC_TF32, qsim.PREC_BF16X3], ids=["tf32", "bf16x3"])
def test_batch_of_both_tensor_core_forms(prec, graph):
    # 4096-amplitude tiles with dense ops of every width the warp-level form takes, beside tcgen05 plans, a plan whose
    # tiles are smaller and one without tensor-core ops
    forms = [(inputs.random_brick(15, 6, 1), 13, 5, 0), (inputs.random_brick(15, 6, 2), 13, 5, 1),
             (inputs.qft_rz_cx(14, 2, 3), 12, 4, 0), (inputs.grover(13, 3, 77), 12, 3, 0), (inputs.ghz(14), 12, 2, 0),
             (inputs.random_brick(12, 6, 4), 8, 5, 0), (inputs.qaoa_maxcut(14, 2, 5), 12, 5, 1)]
    plans = [qsim.plan_stages(c, m=m, inner=2, k=k, eps=1e-3, prec=prec, tcgen05=t, graph=graph, reorder=2, diag_exempt=1)
             for c, m, k, t in forms]
    states, launch = qsim.run_batch(plans)
    assert graph or launch["launches"] == 2
    for (c, m, k, t), p, st in zip(forms, plans, states):
        assert streams_of(st) == streams_of(qsim.run(p)), (c.family, k, t)
        assert st.fidelity(oracle.simulate(c)) >= 0.99
    # no plan without tcgen05 needs the warp-level form: one launch
    states, launch = qsim.run_batch([plans[1], plans[4], plans[5], plans[6]])
    assert graph or launch["launches"] == 1
    for p, st in zip([plans[1], plans[4], plans[5], plans[6]], states):
        assert streams_of(st) == streams_of(qsim.run(p))


def test_run_after_a_refused_batch():
    """A batch is refused after its initial stores are launched; what it allocated may be another run's the moment the
    call returns, on whichever stream: the stores are waited for first."""
    torch = pytest.importorskip("torch")
    c = inputs.random_brick(20, 2, 9)
    kw = dict(m=6, inner=2, k=2, eps=1e-3)
    plan, other = qsim.plan_stages(c, **kw), torch.cuda.Stream()
    wide = qsim.plan_stages(inputs.random_brick(20, 2, 1), m=6, inner=2, k=6, eps=1e-3)
    want = qsim.run(plan).decompress()
    for _ in range(5):
        with pytest.raises(qsim.QsimError) as ei:
            qsim.run_batch([plan, plan, wide])
        assert ei.value.code == qsim.E_INVALID
        assert torch.equal(qsim.run(plan, stream=other).decompress(), want)


def test_batch_bytes_are_its_circuits():
    plans = [qsim.plan_stages(c, m=m, inner=2, k=4, eps=1e-3, mode=qsim.MODE_PERSISTENT)
             for c, m in ((inputs.random_brick(15, 4, 1), 13), (inputs.qft_rz_cx(12, 1, 2), 9))]
    _, launch = qsim.run_batch(plans)
    qsim.profile_enable(True)
    try:
        single = [qsim.run(p).kernel_stats()[launch["name"]] for p in plans]
    finally:
        qsim.profile_enable(False)
    assert launch["alg_bytes"] == sum(s["alg_bytes"] for s in single)
    assert launch["alg_flops"] == sum(s["alg_flops"] for s in single)
