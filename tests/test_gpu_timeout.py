"""Failure path of the persistent kernels that plain calls use: a cross-CTA wait that can never end (test hook) runs out after two to
three seconds, the call returns WIND_ERR_TIMEOUT and says which wait it was, and the next call on the context is right.  (The kernels
with grid barriers and with arrival counters: test_gpu_parity.py.)"""
import numpy as np
import pytest

from naive_model import random_weights
from test_gpu_parity import pkg, ragged_case  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,dtype,B,T,E,P,L,H,V,W,sites", [
    ("CLUSTERS", "bf16", 3, 30, 64, 128, 1, 128, 200, 8, range(50, 66)),      # one slot per cluster
    ("CLUSTERS", "bf16", 60, 30, 64, 640, 1, 640, 200, 8, range(50, 66)),     # eight slots, remainder units, queue
    ("CLUSTERS", "bf16", 128, 40, 64, 256, 1, 256, 200, 32, range(50, 66)),   # the other kernel launched behind them
    ("CLUSTERS", "bf16", 9, 30, 64, 640, 2, 256, 200, 8, range(50, 72)),      # two layers: the recurrent terms' clusters leave too
    ("WIDE", "bf16", 5, 30, 64, 192, 1, 1024, 600, 8, (3, 4)),
    ("GRID", "f32", 4, 24, 160, 320, 1, 300, 500, 8, (5,)),
])
def test_wait_that_never_ends(pkg, name, dtype, B, T, E, P, L, H, V, W, sites):  # noqa: F811
    S = 3
    w, enc, lens = ragged_case(2200 + B, B=B, T=T, D=64, E=E, P=P, L=L, H=H, V=V, bias=3.0, dtype=dtype)
    lens = np.sort(lens)[::-1].astype(np.int32) // (4 if B > 100 else 1)      # short but for one: the lengths favour clusters
    lens[0] = T
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    d = model.device
    enc_d, lens_d = pkg.to_device_enc(model, enc), torch.from_numpy(lens).to(d)
    tok = torch.full((B, T * S), -1, dtype=torch.int32, device=d)
    frm, olen = tok.clone(), torch.zeros(B, dtype=torch.int32, device=d)
    ws = pkg.alloc_workspace(model, B, T, W)

    def decode():
        return pkg.wind_decode_greedy(model, enc_d, lens_d, W, S, tok, frm, olen, ws, check=False)

    assert decode() == 0
    assert pkg.binding.wind_debug_loop_kernel(ws) == getattr(pkg.binding, "WIND_LOOP_" + name)
    ref = [x.clone() for x in (tok, frm, olen)]
    prev = pkg.wind_debug_stall_barrier(1)
    try:
        st = decode()
        stats = pkg.wind_read_stats(ws)
    finally:
        pkg.wind_debug_stall_barrier(prev)
    assert st == pkg.binding.WIND_ERR_TIMEOUT and stats["status"] == st
    assert stats["timeout_site"] in sites and 0 <= stats["timeout_cta"] < torch.cuda.get_device_properties(d).multi_processor_count
    tok.fill_(-1), frm.fill_(-1)
    assert decode() == 0
    stats = pkg.wind_read_stats(ws)
    assert stats["timeout_site"] == 0
    for a, b in zip((tok, frm, olen), ref):
        assert torch.equal(a, b)


@pytest.mark.parametrize("prefix_search", [False, True])
def test_beam_search_wait_that_never_ends(pkg, prefix_search):  # noqa: F811
    r = np.random.default_rng(2300)
    w = random_weights(r, 16, 32, 64, 1, 64, 100, act=0, blank_bias=2.5, bias_scale=0.1)
    w["dtype"] = "f32"
    model = pkg.WindModel(w)
    enc = r.standard_normal((20, 16)).astype(np.float32)
    ref = pkg.wind_beam_search(model, enc, 4, 3, 3, prefix_search=prefix_search)
    prev = pkg.wind_debug_stall_barrier(1)
    try:
        out = pkg.wind_beam_search(model, enc, 4, 3, 3, check=False, prefix_search=prefix_search)
    finally:
        pkg.wind_debug_stall_barrier(prev)
    assert out[2] == pkg.binding.WIND_ERR_TIMEOUT
    again = pkg.wind_beam_search(model, enc, 4, 3, 3, prefix_search=prefix_search)
    assert again[2] == 0 and again[1] == ref[1] and len(again[0]) == len(ref[0])
    for a, b in zip(again[0], ref[0]):
        assert list(a[0]) == list(b[0]) and list(a[1]) == list(b[1]) and a[2] == b[2]
