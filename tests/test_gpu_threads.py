"""Host threads: a decode as the first thing a thread does on the GPU (no context is current in it yet), on the default stream and on
another thread's stream, and several threads at once, each on a stream of its own."""
import threading

import numpy as np
import pytest

from test_gpu_parity import pkg, ragged_case  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Prepared:
    def __init__(self, pkg, seed, W, S=3, **dims):  # noqa: F811
        w, enc, lens = ragged_case(seed, bias=3.0, dtype="bf16", **dims)
        B, T = dims["B"], dims["T"]
        self.pkg, self.W, self.S = pkg, W, S
        self.model = pkg.WindModel(w)
        self.enc, self.lens = pkg.to_device_enc(self.model, np.nan_to_num(enc)), torch.from_numpy(lens).to(self.model.device)
        self.out = [torch.full((B, T * S), -1, dtype=torch.int32, device=self.model.device) for _ in range(2)]
        self.out.append(torch.zeros(B, dtype=torch.int32, device=self.model.device))
        self.ws = pkg.alloc_workspace(self.model, B, T, W)

    def decode(self, stream):
        return self.pkg.wind_decode_greedy(self.model, self.enc, self.lens, self.W, self.S, *self.out, self.ws, stream=stream, check=False)


SHAPES = [dict(B=5, T=30, D=64, E=64, P=128, L=1, H=128, V=200), dict(B=128, T=30, D=64, E=64, P=256, L=1, H=256, V=300),
          dict(B=6, T=30, D=64, E=64, P=128, L=2, H=128, V=200), dict(B=8, T=30, D=64, E=64, P=128, L=1, H=1024, V=600)]


def in_threads(jobs):
    got = [None] * len(jobs)

    def run(i):
        got[i] = jobs[i]()

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return got


@pytest.mark.parametrize("which", range(len(SHAPES)))
def test_first_call_of_a_thread(pkg, which):  # noqa: F811
    one = Prepared(pkg, 2400 + which, 8, **SHAPES[which])
    here = torch.cuda.Stream()
    assert one.decode(here) == 0
    ref = [x.clone() for x in one.out]
    torch.cuda.synchronize()
    for stream in (torch.cuda.default_stream(), here):
        assert in_threads([lambda: one.decode(stream)]) == [0]
        for a, b in zip(one.out, ref):
            assert torch.equal(a, b)


def test_threads_with_a_stream_each(pkg):  # noqa: F811
    all_ = [Prepared(pkg, 2400 + i, 8, **s) for i, s in enumerate(SHAPES)]
    streams = [torch.cuda.Stream() for _ in all_]
    assert [a.decode(s) for a, s in zip(all_, streams)] == [0] * len(all_)
    refs = [[x.clone() for x in a.out] for a in all_]
    torch.cuda.synchronize()
    for k in range(len(all_)):
        all_[k].out[2].zero_()
    torch.cuda.synchronize()
    got = in_threads([(lambda a=a, s=s: [a.decode(s) for _ in range(20)]) for a, s in zip(all_, streams)])
    assert got == [[0] * 20] * len(all_)
    for a, ref in zip(all_, refs):
        for x, y in zip(a.out, ref):
            assert torch.equal(x, y)
