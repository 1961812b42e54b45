"""The flux rule's number of entering ions, drawn beside the previous step (one 64-ion chunk of the mean
per lane) and, in a run's first step, by the scan: below one chunk, around one, several, and more than
a warp of chunks; equal to the oracle's count in every step."""
import pytest

import oracle
import paper_2205_06557_gb300 as od
from paper_2205_06557_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mean", [0.5, 40.0, 64.0, 65.0, 300.0, 2500.0])
def test_entering_ions_equal_the_oracle(mean):
    p = W.tiny()
    p.update(R=4e-4, H=1e-3, dust=[], nu=0.0, n_ions=0, flags=od.F_FLUX_INJECT | od.F_NO_IONION | od.F_NO_EOUT)
    o = oracle.Oracle(dict(p, n_ions=1, oracle_flags=oracle.F_FLUX_INJECT))
    p["dt"] *= mean / (sum(o.injections(s) for s in range(1, 401)) / 400)  # the mean grows with the time step
    o = oracle.Oracle(dict(p, n_ions=1, oracle_flags=oracle.F_FLUX_INJECT))
    run = od.Run(p)
    run.step(6)
    _, ev = run.series(1, 6)
    run.close()
    assert [int(e) for e in ev[:, 9:12].sum(1)] == [o.injections(s) for s in range(1, 7)]
