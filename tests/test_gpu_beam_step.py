"""The beam search's iteration as one kernel, at the sizes where its split can go wrong, against the oracle: rows that are no
multiple of 32, more updates than a pass takes, joint rows in several passes, every length of a thread's list of best entries."""
import numpy as np
import pytest

import oracle
from naive_model import random_weights
from test_gpu_beam import pkg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,P,L,H,V,act,W,K,S", [
    (8, 8, 1, 8, 6, 0, 1, 1, 2),            # less of everything than SMs
    (24, 40, 2, 56, 35, 1, 5, 5, 3),        # two layers, tails of rows, two passes of updates
    (40, 24, 1, 160, 150, 0, 64, 8, 2),     # more labels than SMs, 512 joint rows in several passes, widest window
    (32, 184, 1, 64, 449, 1, 3, 16, 2),     # widest beam, two hidden units in some CTAs
    (20, 24, 1, 32, 30, 0, 4, 3, 3),        # rows that are no multiple of eight: the per-phase kernels
])
def test_beam_iteration_kernel(pkg, E, P, L, H, V, act, W, K, S):  # noqa: F811
    decided = 0
    for seed in range(6):
        r = np.random.default_rng(9000 + 10 * seed + K)
        w = random_weights(r, 16, E, P, L, H, V, act=act, blank_bias=2.5, bias_scale=0.1)
        w["dtype"] = "f32"
        T = int(r.integers(8, 14))
        enc = r.standard_normal((T, 16)).astype(np.float32)
        want, gap, steps = oracle.beam_search(oracle.Model(w), enc, T, W, K, S, max_hyps=256)
        got, gsteps, st = pkg.wind_beam_search(pkg.WindModel(w), enc, W, K, S, max_hyps=256)
        assert st == 0 and len(got) >= 1
        assert abs(got[0][2] - want[0][2]) < 1e-3
        if gap < 2e-5:
            continue
        decided += 1
        a = {tuple(int(x) for x in h[0]): h for h in want}
        b = {tuple(int(x) for x in h[0]): h for h in got}
        assert gsteps == steps and set(a) == set(b)
        assert all(abs(a[k][2] - b[k][2]) < 1e-4 and list(a[k][1]) == list(b[k][1]) for k in a)
    print(f"[beam iteration] K={K} W={W}: {decided}/6 cases decidable and equal to the oracle")
    assert decided >= (1 if K < 8 else 0)
