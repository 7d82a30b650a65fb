"""FP64 angular step with J blocks of very different size.

Nothing mixes the blocks of different J, so each keeps its own relative accuracy however small it is:
the bound of the two forms' difference (1e-13, see test_gpu_f64tc.py) holds block by block."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng,ne", [(40, 1), (31, 2), (180, 1)])
def test_every_J_keeps_its_relative_accuracy(ng, ne):
    from paper_2412_10167_gb300 import mw3
    cfg = W.shrunk(W.C3 if ne == 2 else W.C2, "f64s", NR=24, nr=20, ngamma=ng, J=[0, 1, 3], omega_max=2,
                   nE=8, kmin=0, vmax=-1, E_hi_eV=0.5, products=None)
    out = []
    for form in (0, 1):
        pr = mw3.Propagator(cfg, precision="fp64", tuning=dict(f64_tc=form))
        q = W.random_unit_state(pr.shape, 9)
        n = [(min(J, 2) + 1) * ne for J in cfg["J"]]
        assert sum(n) == pr.shape[0]
        cut = np.cumsum([0] + n)
        for i, s in enumerate((1e-30, 1.0, 1e-15)):
            q[cut[i]:cut[i + 1]] *= s
        out.append(pr.apply_hs(q).reshape(pr.shape))
        pr.close()
    for a, b in zip(cut[:-1], cut[1:]):
        ref = out[0][a:b]
        assert np.linalg.norm(ref) > 0
        assert np.linalg.norm(out[1][a:b] - ref) <= 1e-13 * np.linalg.norm(ref)
