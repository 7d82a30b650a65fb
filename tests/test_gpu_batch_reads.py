"""Probability reads of a J in a batch against the same J alone, bit for bit.

The grid is large enough for a J's flux sum to be cut differently if the cut depended on the batch
(6,600 points of J = 10, 64 energies), and the J differ in their number of points. Reads after a
flush and with pending energy-ring slots, which are summed by kernels of their own."""
import copy

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_batched_J_reads_equal_single_J_bitwise(precision):
    from paper_2412_10167_gb300 import mw3
    cfg = W.shrunk(W.C2, "batchreads", NR=40, nr=36, ngamma=20, J=[10, 9, 8, 7, 6, 5, 4, 3, 2, 1],
                   omega_max=10, nE=64, kmin=0, products=None)
    kb = 8

    def reads(c):
        pr = mw3.Propagator(c, precision=precision, tuning=dict(kb=kb))
        out = []
        for n in (3, 2 * kb - 3, 5):         # pending slots alone, flushed sums, both
            pr.propagate(n)
            out += pr.probabilities()[1:]
        pr.close()
        return out

    batch = reads(cfg)
    for iJ in (0, 4, 9):
        one = copy.deepcopy(cfg)
        one["J"] = [cfg["J"][iJ]]
        for b, s in zip(batch, reads(one)):
            assert np.array_equal(s[0], b[iJ])
