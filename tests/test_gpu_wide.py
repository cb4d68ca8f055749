"""The resident kernel for large vocabularies: a vocabulary tile's remainder, one and several row groups, windows evaluated in
parts, every box size of the state, slots by length.  Transcripts and all counters (which are kept per window) must be those of
the kernel with streamed weights, transcripts those of the oracle under the rule of the parity tests."""
import numpy as np
import pytest

from test_gpu_parity import check_against_oracle, pkg, ragged_case  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,D,E,P,H,V,act,W,S", [
    (1, 40, 64, 64, 64, 1024, 130, 1, 16, 3),       # one utterance, one K block of the state, two entries in the second tile
    (5, 30, 64, 64, 192, 1024, 127, 0, 64, 2),      # widest window, 51 rows of it at a time at first; three K blocks
    (16, 24, 64, 64, 256, 1024, 600, 1, 16, 10),    # exactly two row groups
    (17, 24, 64, 64, 128, 1024, 600, 0, 16, 1),     # 15 rows of a window of 16 at a time
    (64, 40, 64, 64, 64, 1024, 300, 1, 8, 4),       # most utterances, four rows at a time
    (33, 20, 64, 128, 320, 1024, 1000, 0, 1, 5),    # window of one frame, 64-row state box
    (9, 24, 64, 64, 1024, 640, 8000, 0, 16, 3),     # ten K blocks: the last stage of z is cut short, one accumulator
    (3, 24, 64, 64, 512, 896, 10000, 0, 10, 2),     # fourteen, two of them in shared memory; boxes of 32 and 16 rows
    (33, 20, 64, 64, 512, 192, 10000, 0, 32, 3),    # three K blocks: boxes longer than the operand
    (20, 20, 64, 64, 512, 1344, 3000, 1, 8, 3),     # twenty-one, nine of them in shared memory: one stage of 64 KB
])
def test_large_vocabulary_kernel(pkg, B, T, D, E, P, H, V, act, W, S):  # noqa: F811
    w, enc, lens = ragged_case(1500 + B + P, B=B, T=T, D=D, E=E, P=P, L=1, H=H, V=V, act=act, blank_id=0 if B % 2 else None,
                               bias=3.0, dtype="bf16")
    if B > 4:
        lens[2] = 0
    model = pkg.WindModel(w)
    got = pkg.decode(model, enc, lens, W, S)
    pkg.binding.wind_set_loop_options(resident=False)
    try:
        want = pkg.decode(model, enc, lens, W, S)
    finally:
        pkg.binding.wind_set_loop_options()
    for a, b in zip(got[:3], want[:3]):
        assert np.array_equal(a, b)
    for k in ("steps", "joint_rows", "tokens", "forced", "frames", "jump_hist"):
        assert got[3][k] == want[3][k], k
    assert got[3]["tokens"] > 0
    check_against_oracle(pkg, w, enc, lens, W, S, kernels=2, round_bf16=True, margin=2e-2)
