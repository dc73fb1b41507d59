"""Bounds and states at the edge of what the run kernel's lists and strides hold."""
import numpy as np
import pytest

import oracle
import workloads as wl
from tests._compare import assert_same_state

pytestmark = pytest.mark.gpu

itpp = pytest.importorskip("paper_2601_14400_gb300")


# Few strings and one class of magnitudes: a gate doubles the state, and the
# select of a first gate lists every child there is.
@pytest.mark.parametrize("M", [114, 115, 120, 127, 128, 129])
@pytest.mark.parametrize("batch", [False, True])
def test_list_holds_every_child(M, batch):
    # seven commuting strings of angle 3: tanh(3)^7 = 0.966, half an octave holds
    # all of their products
    n = 40
    x = np.zeros((8, 1), dtype=np.uint64)
    z = (np.uint64(1) << np.arange(8, dtype=np.uint64))[:, None]
    H = wl.Hamiltonian(n, x, z, np.full(8, 3.0))
    o = oracle.Oracle(n, x, z, H.alpha, 1.0, 0.0, M, 1)
    o.apply_layers(2)
    if batch:
        p = itpp.BatchPropagator([H, H], 1.0, 0.0, M, 1, table_load_pct=50)
        p.apply_trotter_layer(2)
        got = p.terms(1)
    else:
        p = itpp.Propagator(n, x, z, H.alpha, 1.0, 0.0, M, 1)
        p.apply_trotter_layer(2)
        got = p.terms()
    assert_same_state(got, o.terms(), f"M {M}")
