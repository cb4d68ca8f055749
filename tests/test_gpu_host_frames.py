"""How the host entry point brings the frames over: page-locked memory by one kernel (whole 16-byte pieces, several chunks per
utterance), page-locked memory of odd frames and pageable memory by copies.  The transcripts are those of the device entry point."""
import numpy as np
import pytest

from test_gpu_parity import pkg, ragged_case  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,pinned,offset", [(8, True, 0), (256, True, 0), (256, False, 0), (6, True, 0), (8, True, 1)])
def test_frames_from_the_host(pkg, D, pinned, offset):  # noqa: F811
    B, T, W, S = 5, 70, 4, 3
    w, enc, lens = ragged_case(1700 + D + offset, B=B, T=T, D=D, E=16, P=16, L=1, H=16, V=20)
    model = pkg.WindModel(w)
    want = pkg.decode(model, enc, lens, W, S)
    max_out = want[0].shape[1]
    flat = torch.zeros(B * T * D + offset, dtype=torch.float32)        # offset: a start off the 16-byte grid
    flat = flat.pin_memory() if pinned else flat
    enc_h = flat[offset:].view(B, T, D)
    enc_h.copy_(torch.from_numpy(enc))
    len_h = torch.from_numpy(lens)
    tok, frm = torch.full((B, max_out), -1, dtype=torch.int32), torch.full((B, max_out), -1, dtype=torch.int32)
    olen = torch.zeros(B, dtype=torch.int32)
    ws = pkg.alloc_workspace(model, B, T, W, host_staging_max_out=max_out)
    assert pkg.wind_decode_greedy_host(model, enc_h, len_h, W, S, tok, frm, olen, ws) == 0
    assert np.array_equal(olen.numpy(), want[2])
    for b in range(B):
        assert np.array_equal(tok.numpy()[b, :olen[b]], want[0][b, :olen[b]])
        assert np.array_equal(frm.numpy()[b, :olen[b]], want[1][b, :olen[b]])


def test_frames_whose_head_alone_is_page_locked(pkg):  # noqa: F811
    # Two utterances of 64 KB: the first one's pages are registered, the second one's are not, so the GPU can reach the first
    # byte of the array and not the last.  With the second half registered too (a range of its own) the GPU reaches all of it.
    import mmap

    B, T, D, W, S = 2, 64, 256, 4, 3
    w, enc, _ = ragged_case(1790, B=B, T=T, D=D, E=16, P=16, L=1, H=16, V=20)
    enc = np.nan_to_num(enc)
    lens = np.array([T, T - 3], dtype=np.int32)
    model = pkg.WindModel(w)
    want = pkg.decode(model, enc, lens, W, S)
    max_out = want[0].shape[1]
    half = T * D * 4
    assert half % mmap.PAGESIZE == 0
    area = mmap.mmap(-1, B * half)
    enc_h = torch.frombuffer(area, dtype=torch.float32).view(B, T, D)
    enc_h.copy_(torch.from_numpy(enc))
    rt = torch.cuda.cudart()
    registered = []
    ws = pkg.alloc_workspace(model, B, T, W, host_staging_max_out=max_out)
    try:
        for part in range(B):
            assert int(rt.cudaHostRegister(enc_h.data_ptr() + part * half, half, 0)) == 0
            registered.append(enc_h.data_ptr() + part * half)
            tok, frm = torch.full((B, max_out), -1, dtype=torch.int32), torch.full((B, max_out), -1, dtype=torch.int32)
            olen = torch.zeros(B, dtype=torch.int32)
            assert pkg.wind_decode_greedy_host(model, enc_h, torch.from_numpy(lens), W, S, tok, frm, olen, ws) == 0
            assert np.array_equal(olen.numpy(), want[2])
            for b in range(B):
                assert np.array_equal(tok.numpy()[b, :olen[b]], want[0][b, :olen[b]])
                assert np.array_equal(frm.numpy()[b, :olen[b]], want[1][b, :olen[b]])
    finally:
        torch.cuda.synchronize()
        for at in registered:
            rt.cudaHostUnregister(at)
