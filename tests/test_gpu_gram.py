"""The tensor-core measurement at the edges of its work units: sizes with one short tile, one
super-tile, ragged super-tiles, several replicas per pass of the line-order copies, and rows of one to
ten words.  Records are integers, so every comparison is exact."""
import numpy as np
import pytest

import oracle
from paper_2305_12161_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    from paper_2305_12161_gb300 import ising as m
    m.lib()
    return m


@pytest.mark.parametrize("L", [64, 128, 192])
def test_record_equals_oracle(ising, L):
    states = [inputs.neel_state(L), inputs.stripe_state(L, 8, "y"), inputs.uniform_state(L, 1),
              inputs.uniform_state(L, -1), inputs.random_state(L, 5), inputs.random_state(L, 6, 0.9)]
    with ising.Ising(L, replicas=len(states), seed=1) as q:
        for r, s in enumerate(states):
            q.set_spins(s, r)
        rec = q.measure()
    for r, s in enumerate(states):
        assert np.array_equal(rec[r], oracle.record(s, 0)), r


@pytest.mark.parametrize("L,R", [(64, 33), (256, 3), (320, 2), (384, 1), (448, 1), (512, 6), (576, 1), (640, 2),
                                 (768, 1)])
def test_record_equals_bit_counts(ising, L, R):
    with ising.Ising(L, replicas=R, seed=11) as a, \
            ising.Ising(L, replicas=R, seed=11, corr=ising.CORR_POPCOUNT) as b:
        for n in (0, 5):
            a.sweep(n)
            b.sweep(n)
            assert np.array_equal(a.measure(), b.measure()), n


@pytest.mark.parametrize("L,R", [(512, 1), (768, 2), (1024, 1), (1280, 1)])
def test_line_order_units_equal_bit_counts(ising, L, R):
    """Sizes of whole super-tiles with the line-order copies: diagonal and off-diagonal units follow
    one another on a block, whose A tiles share tensor memory with the other's second accumulator."""
    with ising.Ising(L, replicas=R, seed=23) as a, \
            ising.Ising(L, replicas=R, seed=23, corr=ising.CORR_POPCOUNT) as b:
        for n in (0, 3):
            a.sweep(n)
            b.sweep(n)
            assert np.array_equal(a.measure(), b.measure()), n


@pytest.mark.parametrize("L,R", [(512, 3), (640, 1), (768, 2), (1024, 1)])
def test_without_scratch_equals_bit_counts(ising, L, R):
    """The packed lattice read in place at sizes that otherwise have copies in line order: the x axis
    transposed by the filling warps, A tiles of off-diagonal units in shared memory."""
    with ising.Ising(L, replicas=R, seed=29) as a, \
            ising.Ising(L, replicas=R, seed=29, corr=ising.CORR_POPCOUNT) as b:
        a.measure()
        a.inject_scratch_refusal()
        for n in (0, 3):
            a.sweep(n)
            b.sweep(n)
            l0 = a.launch_count()
            assert np.array_equal(a.measure(), b.measure()), n
            assert a.launch_count() - l0 == 2  # the record's initialisation and the products
