"""bench.py's byte model of the reduced inner solves, against a hand count, and
which screens it is used for."""
from types import SimpleNamespace

import numpy as np
import pytest

from test_bench_host import _bench


def test_reduced_bytes_hand_count():
    """Two scenarios of 2 and 1 outer iterations on a matrix pair with 9 and 6
    rows and 25 and 15 factor entries (FP64 vectors, w = 8): per outer iteration
    and matrix one forward and one backward pass that read and write the vector
    once (4 w bytes a row) and read the factor with its column indices twice."""
    b = _bench()
    info = dict(n_p=9, n_q=6, nnz_p=30, nnz_q=20, nnz_lp=25, nnz_lq=15)
    iters = np.array([[2, 3, 4], [1, 2, 0]], dtype=np.int32)
    n_bus, n_branch, w = 10, 14, 8
    vec = 3 * 4 * w * (9 + 6)
    mats = 3 * 2 * (25 + 15) * (w + 4) / 2  # shared by the two scenarios
    mis = 32 * n_bus * (5 + 3)
    flows = 2 * (16 * n_bus + 8 * n_branch)
    assert b.algorithmic_bytes(info, iters, w, n_bus, n_branch, True) == pytest.approx(
        vec + mats + mis + flows, rel=0, abs=1e-9)


def test_which_screens_are_reduced():
    """At the bench's 1e-4 p.u. only FP64 inner solves with the complete factor."""
    b = _bench()
    for precision in ("fp32", "fp64", "fp16f"):
        for precond in ("exact", "ic0", "jacobi"):
            a = SimpleNamespace(precision=precision, precond=precond)
            assert b.reduced_solves(a) == ((precision, precond) == ("fp64", "exact"))
