"""The persistent loop of the plain-ALU path: its two forms (decoder inside one SM, decoder spread over the grid), rows that
are and are not multiples of four and of 32, weights resident and not, against the oracle under the rule of the parity tests."""
import numpy as np
import pytest

from test_gpu_parity import check_against_oracle, pkg, ragged_case  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B,T,D,E,P,L,H,V,act,W,S", [
    ("f32", 1, 60, 64, 64, 64, 1, 64, 32, 0, 4, 5),        # one SM, one utterance
    ("f32", 150, 20, 20, 24, 24, 2, 40, 30, 1, 3, 2),      # one SM, more utterances than SMs, two layers
    ("f32", 5, 30, 17, 19, 21, 1, 33, 29, 0, 9, 3),        # one SM, rows padded to four, window of more than eight rows
    ("f32", 3, 20, 20, 64, 32, 1, 16, 900, 0, 4, 3),       # one SM, embedding table in L2, more labels than threads
    ("f32", 2, 90, 16, 16, 16, 1, 16, 20, 0, 40, 3),       # one SM, window of more than 32 rows
    ("f32", 160, 40, 30, 64, 64, 1, 64, 63, 1, 32, 2),     # weights in registers: all of them in use, widest window, more utterances than SMs
    ("f32", 4, 30, 9, 1, 33, 1, 64, 1, 0, 17, 3),          # the same, barely: one more unit than half a row, one label, odd window
    ("f32", 4, 30, 9, 65, 64, 1, 64, 63, 0, 8, 3),         # one embedding element too many
    ("bf16", 5, 30, 24, 33, 61, 1, 35, 50, 1, 8, 3),
    ("f32", 9, 24, 32, 160, 320, 1, 300, 500, 0, 8, 4),    # grid: units in some CTAs only, three passes of utterances
    ("f32", 3, 24, 32, 130, 333, 2, 301, 449, 1, 5, 2),    # grid, rows padded to 32, two layers, tanh
    ("f32", 2, 10, 32, 640, 1024, 3, 1024, 4000, 0, 8, 2), # grid, weights too large for the chip
    ("bf16", 6, 24, 40, 24, 40, 2, 56, 35, 0, 4, 3),       # bf16 operands, one SM
    ("bf16", 7, 20, 40, 200, 328, 1, 264, 700, 0, 8, 3),   # bf16 operands, grid
])
def test_persistent_plain_alu_loop(pkg, dtype, B, T, D, E, P, L, H, V, act, W, S):  # noqa: F811
    w, enc, lens = ragged_case(1200 + B + P, B=B, T=T, D=D, E=E, P=P, L=L, H=H, V=V, act=act, blank_id=0 if B % 2 else None,
                               bias=1.5, dtype=dtype)
    rep, out = check_against_oracle(pkg, w, enc, lens, W, S, kernels=1, round_bf16=dtype == "bf16", margin=5e-3)
    assert rep["stats"]["kernels"] == 1
    again = pkg.decode(pkg.WindModel(w), enc, lens, W, S) if dtype == "f32" else None
    if again is not None:
        for a, b in zip(again[:3], out):
            assert np.array_equal(a, b)
