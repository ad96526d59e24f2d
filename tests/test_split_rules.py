"""CPU check that split_rules.py, by which the GPU tests pick the sizes where the sweeps'
split changes, states the rules of the header."""
import ctypes

import numpy as np

import split_rules


def test_restated_rules_are_the_headers(tmp_path):
    lib = ctypes.CDLL(split_rules.compile_rules(str(tmp_path)))
    lib.slots.restype = ctypes.c_longlong
    rng = np.random.default_rng(1)
    totals = [5, 126, 127, 128, 129, 409200, 612863, 612864, 612865, 4902912, 10 ** 9]
    for total in totals + [int(v) for v in np.exp(rng.uniform(2, 20, 500))]:
        assert lib.slots(ctypes.c_longlong(total)) == 128 * split_rules.chunks_per_block(total) - 2
    for _ in range(500):
        plane, n = int(np.exp(rng.uniform(1.1, 12))), int(np.exp(rng.uniform(1.1, 7)))
        for fp64 in (True, False):
            assert lib.segment(ctypes.c_longlong(plane * n), n, int(fp64)) == split_rules.segment(plane, n, fp64)
