"""Which of two kernels decodes is decided on the device, from the lengths: batches around the point where the kernel with grid
barriers takes over from the clusters.  Either way the transcripts and counters are those of the kernel with grid barriers."""
import numpy as np
import pytest

from test_gpu_parity import pkg, ragged_case  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,W,lo", [(113, 8, 30), (113, 8, 3), (128, 16, 30), (112, 5, 30), (128, 16, 1), (90, 12, 25)])
def test_kernel_chosen_by_the_lengths(pkg, B, W, lo):  # noqa: F811
    T, S = 30, 3
    w, enc, lens = ragged_case(1900 + B + W + lo, B=B, T=T, D=64, E=64, P=128, L=1, H=128, V=200, bias=3.0, dtype="bf16")
    r = np.random.default_rng(B + lo)
    lens = r.integers(lo, T + 1, size=B).astype(np.int32)
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    got = pkg.decode(model, enc, lens, W, S)
    pkg.binding.wind_set_loop_options(dataflow=0)
    try:
        want = pkg.decode(model, enc, lens, W, S)
    finally:
        pkg.binding.wind_set_loop_options()
    for a, b in zip(got[:3], want[:3]):
        assert np.array_equal(a, b)
    for k in ("tokens", "forced", "frames", "joint_rows", "jump_hist"):
        assert got[3][k] == want[3][k], k
    assert got[3]["tokens"] > 0


@pytest.mark.parametrize("N,B,W", [(400, 128, 16), (400, 128, 8)])
def test_refilled_rows_either_way(pkg, N, B, W):  # noqa: F811
    T, S = 12, 3
    w, enc, _ = ragged_case(1950 + W, B=N, T=T, D=64, E=64, P=128, L=1, H=128, V=200, bias=3.0, dtype="bf16")
    lens = np.random.default_rng(W).integers(6, T + 1, size=N).astype(np.int32)
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    got = pkg.decode_refill(model, enc, lens, B, W, S)
    pkg.binding.wind_set_loop_options(dataflow=0)
    try:
        want = pkg.decode_refill(model, enc, lens, B, W, S)
    finally:
        pkg.binding.wind_set_loop_options()
    for a, b in zip(got[:3], want[:3]):
        assert np.array_equal(a, b)
