"""Which of two kernels decodes is decided on the device, from the lengths: batches around the point where the kernel with grid
barriers takes over from the clusters.  Either way the transcripts and counters are those of the kernel with grid barriers."""
import numpy as np
import pytest

from conftest import set_loop_mode
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


def loop_kernel_of(pkg, model, enc, lens, W, S):  # noqa: F811
    """Transcripts on device buffers of this test's own, and which kernel's they are."""
    B, T, _ = enc.shape
    d = model.device
    tok, frm = torch.full((B, T * S), -1, dtype=torch.int32, device=d), torch.full((B, T * S), -1, dtype=torch.int32, device=d)
    olen = torch.zeros(B, dtype=torch.int32, device=d)
    ws = pkg.alloc_workspace(model, B, T, W)
    st = pkg.wind_decode_greedy(model, pkg.to_device_enc(model, enc), torch.from_numpy(lens).to(d), W, S, tok, frm, olen, ws)
    assert st == 0
    return pkg.binding.wind_debug_loop_kernel(ws), [x.cpu().numpy() for x in (tok, frm, olen)]


@pytest.mark.parametrize("B,W,T,lo,dim,want", [
    (128, 8, 60, 60, 640, "BARRIERS"),      # equal lengths: three rounds of slots
    (128, 8, 60, 2, 640, "CLUSTERS"),       # ragged ones
    (112, 8, 60, 60, 128, "CLUSTERS"),      # two rounds
    (16, 8, 60, 60, 128, "CLUSTERS"),       # one round
    (128, 32, 60, 60, 128, "BARRIERS"),     # widest window: ten rounds
    (128, 17, 60, 60, 640, "BARRIERS"),
    (64, 32, 60, 60, 128, "COUNTERS"),      # up to 64 rows the other kernel is the one with arrival counters
    (64, 32, 60, 2, 128, "CLUSTERS"),
    (57, 16, 300, 290, 640, "COUNTERS"),
    (28, 16, 60, 60, 640, "CLUSTERS"),
    (400, 24, 100, 100, 640, "STREAMING"),  # more rows than the resident kernels take: the shapes decide
    (400, 24, 100, 10, 640, "STREAMING"),
])
def test_which_kernel_decodes(pkg, B, W, T, lo, dim, want):  # noqa: F811
    S = 3
    w, enc, _ = ragged_case(1980 + B + W + lo, B=B, T=T, D=64, E=64, P=dim, L=1, H=dim, V=200, bias=3.0, dtype="bf16")
    lens = np.random.default_rng(B + lo).integers(lo, T + 1, size=B).astype(np.int32)
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    kernel, got = loop_kernel_of(pkg, model, enc, lens, W, S)
    assert kernel == getattr(pkg.binding, "WIND_LOOP_" + want)
    set_loop_mode(pkg, "barriers")
    kernel, ref = loop_kernel_of(pkg, model, enc, lens, W, S)
    assert kernel == (pkg.binding.WIND_LOOP_STREAMING if want == "STREAMING" else pkg.binding.WIND_LOOP_BARRIERS)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("L,B,W,T,lo,dim,want", [
    (1, 36, 20, 150, 146, 384, "CLUSTERS"),     # three rounds of slots, and still ahead: 0.84 ms against 0.97
    (1, 64, 12, 150, 146, 512, "CLUSTERS"),     # 0.82 against 0.97
    (2, 41, 8, 150, 146, 640, "CLUSTERS"),      # one utterance more than slots: 0.94 against 1.28
    (2, 128, 8, 60, 60, 512, "BARRIERS"),       # equal lengths: four rounds
    (2, 128, 8, 60, 2, 512, "CLUSTERS"),        # ragged ones
    (2, 64, 32, 60, 60, 128, "BARRIERS"),       # widest window: seven rounds
])
def test_which_kernel_decodes_near_the_line(pkg, L, B, W, T, lo, dim, want):  # noqa: F811
    w, enc, _ = ragged_case(1970 + B + W + lo, B=B, T=T, D=64, E=64, P=dim, L=L, H=dim, V=200, bias=3.0, dtype="bf16")
    lens = np.random.default_rng(B + lo).integers(lo, T + 1, size=B).astype(np.int32)
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    kernel, got = loop_kernel_of(pkg, model, enc, lens, W, 3)
    assert kernel == getattr(pkg.binding, "WIND_LOOP_" + want)
    set_loop_mode(pkg, "barriers")
    kernel, ref = loop_kernel_of(pkg, model, enc, lens, W, 3)
    assert kernel == pkg.binding.WIND_LOOP_BARRIERS
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("N,B,W,lo,want", [
    (384, 128, 16, 100, "BARRIERS"),        # rows refilled in the other kernel as well
    (300, 64, 8, 1, "CLUSTERS"),
    (4200, 128, 32, 1, "BARRIERS"),         # more utterances than are put in order or played through
])
def test_which_kernel_refills(pkg, N, B, W, lo, want):  # noqa: F811
    T, S = (100, 3) if N < 1000 else (4, 3)
    w, enc, _ = ragged_case(1990 + N, B=N, T=T, D=64, E=64, P=128, L=1, H=128, V=200, bias=3.0, dtype="bf16")
    lens = np.random.default_rng(N).integers(lo, T + 1, size=N).astype(np.int32)
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    d = model.device
    tok, frm = torch.full((N, T * S), -1, dtype=torch.int32, device=d), torch.full((N, T * S), -1, dtype=torch.int32, device=d)
    olen = torch.zeros(N, dtype=torch.int32, device=d)
    ws = torch.empty(pkg.binding.wind_refill_workspace_bytes(model, N, T, B, W) + 256, dtype=torch.uint8, device=d)
    st = pkg.binding.wind_decode_greedy_refill(model, pkg.to_device_enc(model, enc), torch.from_numpy(lens).to(d), B, W, S, tok, frm, olen, ws)
    assert st == 0 and pkg.binding.wind_debug_loop_kernel(ws) == getattr(pkg.binding, "WIND_LOOP_" + want)
    set_loop_mode(pkg, "barriers")
    want_out = pkg.decode_refill(model, enc, lens, B, W, S)
    for a, b in zip((tok, frm, olen), want_out[:3]):
        assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("B,W,dim,want", [(7, 8, 128, 4), (60, 8, 128, 5), (128, 8, 640, 7), (400, 24, 640, 4)])
def test_launch_count(pkg, B, W, dim, want):  # noqa: F811
    # init, projection, gate table, loop; with more utterances than slots their order; where the lengths decide, the choice and the
    # other kernel; from the host, the kernel that fetches the frames
    T, S = 100, 3
    w, enc, lens = ragged_case(2100 + B, B=B, T=T, D=64, E=64, P=dim, L=1, H=dim, V=200, bias=3.0, dtype="bf16")
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    assert pkg.decode(model, enc, lens, W, S)[3]["launches_setup"] == want
    max_out = T * S
    enc_h, len_h = torch.from_numpy(enc).to(torch.bfloat16).pin_memory(), torch.from_numpy(lens).pin_memory()
    tok = torch.full((B, max_out), -1, dtype=torch.int32)
    ws = pkg.alloc_workspace(model, B, T, W, host_staging_max_out=max_out)
    assert pkg.wind_decode_greedy_host(model, enc_h, len_h, W, S, tok, tok.clone(), torch.zeros(B, dtype=torch.int32), ws) == 0
    assert pkg.wind_read_stats(ws)["launches_setup"] == want + 1
    set_loop_mode(pkg, "barriers")
    assert pkg.decode(model, enc, lens, W, S)[3]["launches_setup"] == 4
