"""The cluster kernel of the decoding loop (models of one or two layers whose decoder fits sixteen CTAs): edges of its tiles.

Every case is decoded in the default mode, which picks the cluster kernel for these shapes (asserted), and with the grid-barrier
kernel; the two use the same arithmetic, so the transcripts must be equal bit for bit, and the first is also checked
against the oracle under the margin rule of the parity tests.
"""
import numpy as np
import pytest

from conftest import set_loop_mode
from test_gpu_choice import loop_kernel_of
from test_gpu_parity import check_against_oracle, pkg, ragged_case  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,P,H,V,act,W,S", [
    (1, 40, 128, 128, 127, 0, 1, 3),       # smallest dimensions, eight vocabulary entries per CTA, one row
    (3, 40, 640, 640, 1024, 0, 8, 10),     # the large model: remainder units, one CTA with eight more labels, one slot per cluster
    (13, 30, 512, 640, 1151, 1, 8, 2),     # no remainder units; 72 labels in every CTA; two slots
    (9, 30, 640, 128, 300, 0, 16, 2),      # padded window of 16
    (25, 24, 256, 384, 1000, 1, 5, 3),     # four slots, six K blocks, odd window
    (28, 42, 512, 640, 552, 1, 1, 3),      # four slots, of which some sit most updates out
    (18, 45, 128, 512, 353, 0, 2, 2),      # three
    (50, 24, 640, 512, 1030, 0, 4, 2),     # eight slots
    (109, 20, 640, 640, 140, 0, 8, 3),     # sixteen slots; some CTAs without a label
    (200, 16, 128, 640, 513, 1, 2, 2),     # more utterances than slots: the queue, longest first
    (40, 20, 384, 256, 200, 0, 32, 3),     # widest window: four slots of 32 rows, refilled
    (17, 20, 640, 640, 1024, 1, 11, 1),    # every emission forces an advance
])
def test_cluster_kernel_edges(pkg, N, T, P, H, V, act, W, S):  # noqa: F811
    w, enc, lens = ragged_case(900 + N + W, B=N, T=T, D=64, E=64, P=P, L=1, H=H, V=V, act=act,
                               blank_id=0 if N % 2 else None, bias=1.5, dtype="bf16")
    rep, out = check_against_oracle(pkg, w, enc, lens, W, S, kernels=2)
    model = pkg.WindModel(w)
    assert loop_kernel_of(pkg, model, enc, lens, W, S)[0] == pkg.binding.WIND_LOOP_CLUSTERS
    set_loop_mode(pkg, "barriers")
    tok, frm, olen, stats, st = pkg.decode(model, enc, lens, W, S)
    assert st == 0 and stats["tokens"] == rep["stats"]["tokens"] and stats["jump_hist"] == rep["stats"]["jump_hist"]
    for a, b in zip((tok, frm, olen), out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("seed,N,T,H,V,W,S", [(8334, 145, 16, 128, 450, 1, 3), (10919, 97, 51, 256, 882, 2, 4), (13837, 189, 55, 384, 619, 8, 2)])
def test_remainder_units_round_like_the_others(pkg, seed, N, T, H, V, W, S):  # noqa: F811
    # Units beyond the first 32 of a CTA are updated by other code than those.  Where it fused the other product of the cell update,
    # one decision of each of these batches came out differently from the kernel with grid barriers.
    w, enc, lens = ragged_case(seed, B=N, T=T, D=64, E=64, P=640, L=1, H=H, V=V, act=0, bias=3.0, dtype="bf16")
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    got = pkg.decode(model, enc, lens, W, S)
    assert loop_kernel_of(pkg, model, enc, lens, W, S)[0] == pkg.binding.WIND_LOOP_CLUSTERS
    set_loop_mode(pkg, "barriers")
    want = pkg.decode(model, enc, lens, W, S)
    for a, b in zip(got[:3], want[:3]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("N,T,P,H,V,act,W,S", [
    (1, 40, 128, 128, 127, 0, 1, 3),       # smallest dimensions, one decoding cluster
    (6, 60, 640, 640, 1024, 0, 4, 10),     # remainder units; two slots in some clusters, one in others
    (13, 30, 512, 640, 1151, 1, 8, 2),     # no remainder units; 72 labels in every CTA; three slots
    (33, 20, 640, 128, 130, 0, 8, 3),      # states that need more shared memory than the decoding CTAs (P far above H), seven slots
    (33, 20, 640, 128, 130, 0, 1, 3),      # the workspace has no room for their exchange: grid barriers
    (9, 30, 640, 128, 300, 0, 16, 2),      # padded window of 16
    (40, 24, 640, 640, 1024, 0, 8, 3),     # all forty slots
    (64, 30, 640, 640, 1024, 0, 8, 10),    # more utterances than slots: the queue, or the other kernel, as the lengths have it
    (60, 16, 256, 384, 1000, 1, 5, 3),
    (25, 20, 384, 256, 200, 0, 32, 3),     # widest window: ten slots, refilled
    (6, 40, 640, 640, 1024, 0, 17, 3),     # padded window of 32 at the largest dimensions: the most shared memory, two slots in some clusters
    (12, 40, 640, 640, 1024, 1, 32, 3),    # and more utterances than slots
    (50, 1, 640, 640, 200, 0, 2, 1),       # utterances of one frame: every update starts afresh
])
def test_two_layer_cluster_edges(pkg, N, T, P, H, V, act, W, S):  # noqa: F811
    w, enc, lens = ragged_case(1300 + N + W, B=N, T=T, D=64, E=64, P=P, L=2, H=H, V=V, act=act,
                               blank_id=0 if N % 2 else None, bias=1.5, dtype="bf16")
    rep, out = check_against_oracle(pkg, w, enc, lens, W, S, kernels=2)
    model = pkg.WindModel(w)
    room = (P, H, W) != (640, 128, 1)
    assert loop_kernel_of(pkg, model, enc, lens, W, S)[0] == (pkg.binding.WIND_LOOP_CLUSTERS if room else pkg.binding.WIND_LOOP_BARRIERS)
    set_loop_mode(pkg, "barriers")
    tok, frm, olen, stats, st = pkg.decode(model, enc, lens, W, S)
    assert st == 0 and stats["tokens"] == rep["stats"]["tokens"] and stats["jump_hist"] == rep["stats"]["jump_hist"]
    for a, b in zip((tok, frm, olen), out):
        assert np.array_equal(a, b)


def test_two_layer_rows_refilled_in_clusters(pkg):  # noqa: F811
    N, T, B, W, S = 150, 14, 32, 4, 3
    w, enc, lens = ragged_case(1400, B=N, T=T, D=64, E=64, P=256, L=2, H=384, V=300, act=0, bias=2.0, dtype="bf16")
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    got = pkg.decode_refill(model, enc, lens, B, W, S)
    ws = torch.empty(pkg.binding.wind_refill_workspace_bytes(model, N, T, B, W) + 256, dtype=torch.uint8, device=model.device)
    tok = torch.full((N, T * S), -1, dtype=torch.int32, device=model.device)
    olen = torch.zeros(N, dtype=torch.int32, device=model.device)
    pkg.binding.wind_decode_greedy_refill(model, pkg.to_device_enc(model, enc), torch.from_numpy(lens).to(model.device), B, W, S, tok, tok.clone(), olen, ws)
    assert pkg.binding.wind_debug_loop_kernel(ws) == pkg.binding.WIND_LOOP_CLUSTERS
    set_loop_mode(pkg, "barriers")
    want = pkg.decode_refill(model, enc, lens, B, W, S)
    for a, b in zip(got[:3], want[:3]):
        assert np.array_equal(a, b)


def test_two_layer_decode_repeated(pkg):  # noqa: F811
    # Small dimensions make short steps and few updates: the recurrent terms' answers come several steps late, over and over.
    w, enc, lens = ragged_case(2402, B=6, T=30, D=64, E=64, P=128, L=2, H=128, V=200, bias=3.0, dtype="bf16")
    enc = np.nan_to_num(enc)
    model = pkg.WindModel(w)
    set_loop_mode(pkg, "barriers")
    want = pkg.decode(model, enc, lens, 8, 3)
    pkg.wind_set_loop_options()
    assert loop_kernel_of(pkg, model, enc, lens, 8, 3)[0] == pkg.binding.WIND_LOOP_CLUSTERS
    for _ in range(60):
        got = pkg.decode(model, enc, lens, 8, 3)
        for a, b in zip(got[:3], want[:3]):
            assert np.array_equal(a, b)
