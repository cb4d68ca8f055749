"""The beam search's iteration as one kernel, at the sizes where its split can go wrong, against the oracle: rows that are no
multiple of 32, more updates than a pass takes, joint rows in several passes, every length of a thread's list of best entries."""
import ctypes

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


@pytest.mark.parametrize("E,P,L,H,V,W,K,S,updates", [
    (640, 640, 1, 96, 200, 32, 16, 2, 12),  # weights that stay beside twelve of the sixteen updates: two passes
    (512, 512, 2, 512, 300, 8, 12, 2, 4),   # two layers beside four updates; joint items of one row group
])
def test_updates_in_passes_beside_resident_weights(pkg, E, P, L, H, V, W, K, S, updates):  # noqa: F811
    plan = pkg.binding.wind_debug_beam_plan(dict(D=16, E=E, P=P, L=L, H=H, V=V), W, K, pkg.binding.WIND_DT_F32, True)[1]
    assert plan["resident"] and plan["updates"] == updates < K
    r = np.random.default_rng(9603 + K)
    w = random_weights(r, 16, E, P, L, H, V, act=0, blank_bias=2.5, bias_scale=0.1)
    w["dtype"] = "f32"
    T = 3
    enc = r.standard_normal((T, 16)).astype(np.float32)
    want, gap, steps = oracle.beam_search(oracle.Model(w), enc, T, W, K, S, max_hyps=256)
    got, gsteps, st = pkg.wind_beam_search(pkg.WindModel(w), enc, W, K, S, max_hyps=256)
    assert st == 0 and gap > 2e-5            # (every pruning is decidable in fp32)
    a, b = ({tuple(int(x) for x in h[0]): h for h in hyps} for hyps in (want, got))
    assert gsteps == steps and set(a) == set(b)
    assert all(abs(a[k][2] - b[k][2]) < 1e-4 and list(a[k][1]) == list(b[k][1]) for k in a)


def search(pkg, model, enc, W, K, S, short):
    """wind_beam_search with a workspace that is `short` bytes smaller: (tokens, frames, lengths, scores, iterations)."""
    L = pkg.load_library()
    T = enc.shape[0]
    dev = pkg.to_device_enc(model, enc[None])[0].contiguous()
    n = ctypes.c_size_t(0)
    assert L.wind_beam_workspace_bytes(model.ref, T, W, K, S, ctypes.byref(n)) == 0
    ws = torch.empty(n.value + 256, dtype=torch.uint8, device="cuda")
    tok, frm = np.full((64, T * S), -1, np.int32), np.full((64, T * S), -1, np.int32)
    ln, sc, nh, steps = np.zeros(64, np.int32), np.zeros(64), ctypes.c_int32(0), ctypes.c_int64(0)
    st = L.wind_beam_search(model.ref, dev.data_ptr(), T, W, K, S, 0, 64, T * S, tok.ctypes.data, frm.ctypes.data, ln.ctypes.data,
                            sc.ctypes.data, ctypes.byref(nh), ctypes.byref(steps), ws.data_ptr() + -ws.data_ptr() % 256, n.value - short,
                            torch.cuda.current_stream().cuda_stream)
    assert st == 0
    return tok, frm, ln, sc, nh.value, steps.value


@pytest.mark.parametrize("dtype,T,E,P,L,H,V,act,W,K,S,bias", [
    ("f32", 40, 24, 40, 1, 56, 35, 0, 1, 4, 3, 1.0),        # lists a frame apart
    ("f32", 9, 16, 24, 2, 40, 60, 1, 8, 3, 2, 1.5),         # most windows cut short by the end of the utterance
    ("f32", 200, 8, 8, 1, 8, 6, 0, 1, 2, 1, 0.0),           # smallest pool of states
    ("bf16", 60, 40, 72, 1, 64, 300, 0, 5, 4, 10, 2.0),     # many rounds of a frame
    ("bf16", 50, 32, 64, 2, 72, 150, 1, 16, 2, 3, 3.0),     # windows longer than the frames ahead
    ("f32", 30, 32, 64, 1, 64, 200, 0, 64, 8, 3, 2.0),      # joint rows in several passes
    ("bf16", 30, 32, 64, 1, 64, 100, 0, 4, 16, 2, 1.0),     # a command has no more rows than the beam
    ("bf16", 60, 640, 640, 1, 640, 1024, 0, 8, 4, 10, 4.0),
    ("f32", 40, 640, 640, 1, 640, 1024, 0, 8, 4, 10, 4.0),  # nothing ahead fits beside the weights
])
def test_evaluating_ahead_changes_nothing(pkg, dtype, T, E, P, L, H, V, act, W, K, S, bias):  # noqa: F811
    r = np.random.default_rng(9700 + T + W)
    w = random_weights(r, 16, E, P, L, H, V, act=act, blank_bias=bias, bias_scale=0.1)
    w["dtype"] = dtype
    model = pkg.WindModel(w)
    enc = r.standard_normal((T, 16)).astype(np.float32)
    for a, b in zip(search(pkg, model, enc, W, K, S, 0), search(pkg, model, enc, W, K, S, 256)):
        assert np.array_equal(a, b)


def test_other_streams_get_their_turn_during_a_search(pkg):  # noqa: F811
    # The resident kernel holds every SM (57 of 64 thousand registers each).  A search of a few hundred milliseconds in one
    # thread, matrix products one after the other on another stream in this one: several of them have to end while the search is
    # still under way.
    import threading
    import time

    w = random_weights(np.random.default_rng(9500), 16, 64, 64, 1, 64, 200, act=0, blank_bias=6.0, bias_scale=0.1)
    w["dtype"] = "f32"
    model = pkg.WindModel(w)
    T, W, K, S = 16000, 1, 4, 2
    enc = np.random.default_rng(9501).standard_normal((T, 16)).astype(np.float32)
    alone = pkg.wind_beam_search(model, enc, W, K, S, max_hyps=K)
    x = torch.zeros(1024, 1024, device="cuda", dtype=torch.bfloat16)
    side, own = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.mm(x, x)
    torch.cuda.synchronize()
    took, result = [], []

    def search():
        with torch.cuda.stream(own):
            t0 = time.perf_counter()
            result.append(pkg.wind_beam_search(model, enc, W, K, S, max_hyps=K))
            took.append((t0, time.perf_counter()))

    thread = threading.Thread(target=search)
    thread.start()
    done = []
    while thread.is_alive():
        with torch.cuda.stream(side):
            torch.mm(x, x)
        side.synchronize()
        done.append(time.perf_counter())
        time.sleep(0.002)
    thread.join()
    t0, t1 = took[0]
    inside = [t for t in done if t0 + 0.3 * (t1 - t0) < t < t0 + 0.9 * (t1 - t0)]
    print(f"[beam turns] search {1e3 * (t1 - t0):.0f} ms, {len(inside)} kernels of another stream in its middle part")
    assert t1 - t0 > 0.1 and len(inside) >= 5
    for a, b in zip(alone[0], result[0][0]):
        assert list(a[0]) == list(b[0]) and list(a[1]) == list(b[1]) and a[2] == b[2]
