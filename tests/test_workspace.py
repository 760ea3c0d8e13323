"""The library-owned workspace: what a call reserves never falls as its shape grows, so that after
the largest call nothing moves, and a graph captured on a workspace that is outgrown later still
finds it."""
import ctypes
import itertools

import numpy as np
import pytest
import torch

# on both sides of every limit of the plans: 32 / 192 / 304 / 1536 / 4096 rows, steps of 20 MB, rows
# of 64 KB and 128 KB, H = 2560
ROWS = [1, 8, 31, 32, 33, 79, 80, 82, 83, 128, 192, 193, 304, 305, 512, 1024, 1375, 1376, 1536, 1537,
        2048, 4095, 4096, 4097, 20000, 65536]
SIZES = [8, 40, 1000, 4096, 4104, 16384, 16392, 20008, 24504, 24576, 24584, 32000, 32768, 32776, 65536,
         65544, 116736, 126464, 131072, 131080, 1 << 20]
HIDDEN = [8, 64, 1024, 2048, 2560, 2568, 4096, 8192]
WIDTH = {0: 2, 1: 4, 2: 2}


@pytest.fixture(scope="module")
def lib(cuda_lib_path):
    lib = ctypes.CDLL(cuda_lib_path)
    i, l, sz = ctypes.c_int, ctypes.c_long, ctypes.c_size_t
    lib.fdllm_workspace_bytes.argtypes, lib.fdllm_workspace_bytes.restype = [i] * 4, sz
    # not in the interface: fdllm::select_reserve_bytes(int64_t rows, int64_t row_bytes),
    # fdllm::lmhead_need_bytes and lmhead_reserve_bytes(int64_t rows, int H, int V)
    for name, sym, args in (("select_reserve", "_ZN5fdllm20select_reserve_bytesEll", [l, l]),
                            ("lm_need", "_ZN5fdllm17lmhead_need_bytesElii", [l, i, i]),
                            ("lm_reserve", "_ZN5fdllm20lmhead_reserve_bytesElii", [l, i, i])):
        f = getattr(lib, sym)
        f.argtypes, f.restype = args, sz
        setattr(lib, name, f)
    return lib


def test_selection_reservation_covers_every_smaller_shape(lib):
    for dtype in WIDTH:
        got = np.array([[lib.select_reserve(r, v * WIDTH[dtype]) for v in SIZES] for r in ROWS])
        need = np.array([[lib.fdllm_workspace_bytes(1, r, v, dtype) for v in SIZES] for r in ROWS])
        assert (got >= need).all()
        assert (np.diff(got, axis=0) >= 0).all() and (np.diff(got, axis=1) >= 0).all()


def test_lmhead_reservation_covers_every_smaller_shape(lib, monkeypatch):
    monkeypatch.delenv("FDLLM_LMHEAD_GEMM", raising=False)
    monkeypatch.delenv("FDLLM_LMHEAD_BN", raising=False)
    shape = (len(ROWS), len(HIDDEN), len(SIZES))
    got, need = np.zeros(shape, np.int64), np.zeros(shape, np.int64)
    for (i, r), (j, h), (k, v) in itertools.product(*map(enumerate, (ROWS, HIDDEN, SIZES))):
        got[i, j, k], need[i, j, k] = lib.lm_reserve(r, h, v), lib.lm_need(r, h, v)
        # the bound that the header states, with its parts' alignment in the header's place
        assert got[i, j, k] <= r * (2 * h + 32 * -(-v // 192) + 12) + 4096
        # enough for the same positions' logits, too
        assert got[i, j, k] >= lib.select_reserve(r, 4 * v)
    assert (got >= need).all()
    for axis in range(3):
        assert (np.diff(got, axis=axis) >= 0).all()


def _captured(call):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.gpu
def test_smaller_calls_leave_the_workspace(fd, monkeypatch):
    """Warm up and capture the largest shape, call smaller ones that need more scratch than it does,
    replay: the workspace has not moved and the results are the first call's."""
    monkeypatch.delenv("FDLLM_LMHEAD_GEMM", raising=False)
    H, V = 2568, 126464
    gen = torch.Generator(device="cuda").manual_seed(4)
    w = (torch.randn(V, H, generator=gen, device="cuda") * H ** -0.5).to(torch.bfloat16)
    h = torch.randn(64, 32, H, generator=gen, device="cuda").to(torch.bfloat16)
    x = torch.randn(64, 32, V, generator=gen, device="cuda").to(torch.bfloat16)
    x_short = x.view(-1)[:64 * 32 * 32000].view(64, 32, 32000)
    mask = (torch.rand(64, 32, generator=gen, device="cuda") < 0.7).to(torch.uint8)
    conf, tok = torch.zeros(64, 32, device="cuda"), torch.zeros(64, 32, dtype=torch.int32,
                                                                device="cuda")

    def lm(B):
        fd.fdllm_lmhead_confidence(h[:B], w, mask[:B], conf[:B], tok[:B])

    def logits(a):
        fd.fdllm_confidence(a, mask, conf, tok)

    for largest, smaller in ((lambda: lm(64), [lambda: lm(48), lambda: lm(43), lambda: lm(6)]),
                             (lambda: logits(x), [lambda: logits(x_short)])):
        for call in (largest, *smaller):  # load every kernel
            call()
        fd.fdllm_release_workspace()
        largest()
        torch.cuda.synchronize()
        first = conf.clone(), tok.clone()
        g = _captured(largest)
        held = _free()
        for call in smaller:
            call()
        assert _free() == held
        conf.zero_(), tok.zero_()
        g.replay()
        torch.cuda.synchronize()
        on = mask != 0
        assert torch.equal(conf[on], first[0][on]) and torch.equal(tok[on], first[1][on])
    assert fd.fdllm_device_status() == 0


@pytest.mark.gpu
def test_graph_on_an_outgrown_workspace(fd):
    """A larger call after the capture: the graph keeps its workspace, results and status word."""
    fd.fdllm_release_workspace()
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(2, 32, 32000, generator=gen, device="cuda").to(torch.bfloat16)
    mask = torch.ones(2, 32, dtype=torch.uint8, device="cuda")
    out = (torch.full((2, 32), -1, dtype=torch.int32, device="cuda"),
           torch.zeros(2, 32, dtype=torch.uint8, device="cuda"),
           torch.zeros(2, dtype=torch.int32, device="cuda"))

    def step():
        fd.fdllm_select(x, mask, 0.75, "profile", *out)

    step()
    torch.cuda.synchronize()
    first = [t.clone() for t in out] + [mask.clone()]
    g = _captured(step)
    big = torch.randn(2000, 32, 1000, generator=gen, device="cuda").to(torch.bfloat16)
    for B in (500, 2000):  # outgrown twice
        fd.fdllm_confidence(big[:B], torch.ones(B, 32, dtype=torch.uint8, device="cuda"))
        mask.fill_(1)
        out[0].fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        for a, b in zip((*out, mask), first):
            assert torch.equal(a, b)
        assert fd.fdllm_device_status() == 0
    x[1, 3, 7] = float("nan")
    mask.fill_(1)
    g.replay()
    assert fd.fdllm_device_status() == fd.ERR_NONFINITE
    assert out[2].tolist()[1] == fd.ROW_NONFINITE
    assert fd.fdllm_device_status() == 0
    fd.fdllm_release_workspace()


@pytest.mark.gpu
def test_call_without_room_during_a_capture(fd):
    """Refused on the host; the capture goes on, and so does the graph."""
    fd.fdllm_release_workspace()
    x = torch.randn(1, 32, 1000, device="cuda").to(torch.bfloat16)
    mask = torch.ones(1, 32, dtype=torch.uint8, device="cuda")
    conf, tok = fd.fdllm_confidence(x, mask)
    big = torch.zeros(100, 32, 8, device="cuda", dtype=torch.bfloat16)
    out = [torch.zeros(100, 32, dtype=t, device="cuda")
           for t in (torch.uint8, torch.float32, torch.int32)]
    c, t = torch.zeros_like(conf), torch.zeros_like(tok)

    def calls():
        with pytest.raises(fd.FdllmError) as e:
            fd.fdllm_confidence(big, *out)
        assert e.value.status == fd.ERR_CUDA
        fd.fdllm_confidence(x, mask, c, t)

    torch.cuda.synchronize()
    g = _captured(calls)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(c, conf) and torch.equal(t, tok)
    fd.fdllm_confidence(big, *out)  # grows now
    assert fd.fdllm_device_status() == 0
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(c, conf) and fd.fdllm_device_status() == 0
