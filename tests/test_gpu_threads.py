"""Runs on several threads whose first launches come at once, in a process of their own: what the library asks of a device
once (SM count, kernel attributes, launch shapes) is asked under whichever thread comes first."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import threading
from paper_2410_14088_gb300 import inputs, qsim

forms = [dict(), dict(k=5), dict(prec=1, k=5, tcgen05=1), dict(prec=1, k=5), dict(prec=2, k=5, tcgen05=1), dict(codec=2),
         dict(mode=1, k=4), dict(mode=1, prec=1, k=5, tcgen05=1), dict(mode=1, k=2, tile_bits=10), dict(mode=1, codec=2)]
plans = [qsim.plan_stages(inputs.random_brick(15, 5, 7), **dict(dict(m=12, inner=2, k=4, eps=1e-3), **f)) for f in forms]
streams = lambda st: [st.block_stream(b) for b in range(8)]
got, start = [None] * len(plans), threading.Barrier(len(plans))


def work(i):
    start.wait()
    got[i] = streams(qsim.run(plans[i]))


threads = [threading.Thread(target=work, args=(i,)) for i in range(len(plans))]
[t.start() for t in threads]
[t.join() for t in threads]
for f, p, g in zip(forms, plans, got):
    assert g is not None and g == streams(qsim.run(p)), f
print("threads ok")
"""


def test_first_launches_on_several_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "threads ok" in r.stdout, r.stdout + r.stderr
