"""Runs of small steps in one launch: which steps share a launch depends on the
number of units, and the results must not.  Circuits whose steps are all small
(one run), mixed with tensor-core steps, and sliced ones, at unit counts on both
sides of each limit, in every kind of precision, bit for bit; the smallest
against the state vector."""
import numpy as np
import pytest

import tn_inputs as I

from _lib import tnlib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["c64", "split_bf16", "scaled_fp16"])
@pytest.mark.parametrize("rows,cols,depth,num_open,num_sliced", [(3, 3, 6, 2, 2), (4, 4, 8, 6, 3), (4, 5, 12, 5, 9)])
def test_unit_count_does_not_change_the_amplitudes(rows, cols, depth, num_open, num_sliced, precision):
    T = tnlib()
    n = rows * cols
    p = T.plan(T.build_network(T.random_circuit(rows, cols, depth, 3), list(range(n - num_open, n))),
               num_sliced=num_sliced, search_trials=8, seed=1)
    words = I.bitstrings(n, 3, 9)
    slices = p.info()["num_slices"]
    ref = None
    for per_group in (1, 2, 64, 512):
        for rows_at_once in (1, 3):  # units per launch: slices of the group x bitstrings of the call
            got = np.concatenate([p.contract_amplitudes(words[i:i + rows_at_once], precision=precision,
                                                        units_per_group=min(per_group, slices))
                                  for i in range(0, 3, rows_at_once)])
            if ref is None:
                ref = got
            assert np.array_equal(got, ref), (per_group, rows_at_once)


def test_single_run_matches_the_state_vector_with_fewer_launches():
    T = tnlib()
    from oracle import circuit as OC
    from oracle import statevector as SV
    n, open_q = 12, [9, 10, 11]
    p = T.plan(T.build_network(T.random_circuit(3, 4, 8, 5), open_q), search_trials=8, seed=1)
    words = I.bitstrings(n, 2, 5)
    got, rep = p.contract_amplitudes(words, precision="c64", report=True)
    got, rep = p.contract_amplitudes(words, precision="c64", report=True)  # (the first call also ran the invariant steps)
    ref = SV.amplitudes(SV.simulate(OC.random_circuit(3, 4, 8, 5), n), n, [I.bits_of(w, n) for w in words], open_q)
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    assert rep["kernel_launches"] < p.info()["num_steps"] / 2, rep["kernel_launches"]
