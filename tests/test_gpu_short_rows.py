"""Short rows (at most 64 KB each, more than 304 of them): the reduction gives each warp a unit
of at most 512 16-byte vectors.  Row lengths on the edges of a lane's batch, of a unit and of
the range, against the oracle at the selection's own bars."""
import ctypes

import numpy as np
import pytest
import torch

import fdllm_synth as syn
import oracle
from gpu_util import check_confidence, check_select

DT = {"bf16": (torch.bfloat16, 8), "fp16": (torch.float16, 8), "fp32": (torch.float32, 4)}


def _rows(dtype, vecs, seed):
    """10 x 32 rows of `vecs` vectors: ordinary ones and, in the first batch row, every kind of
    unusual one that still has a confidence."""
    t, per = DT[dtype]
    w = syn.Workload("short", 10, 32, vecs * per, dtype, 1.0, "target", 0.3, 3.0)
    x = syn.make_logits(w, seed=seed, device="cuda")
    V = vecs * per
    x[0, 0] = torch.finfo(t).min               # every logit the type's lowest: c = 1 / V
    x[0, 1] = -torch.inf                       # only the last logit is finite
    x[0, 1, V - 1] = 1.0
    x[0, 2, [0, V - 1]] = 30.0                 # a tie across the row (its units): index 0
    x[0, 3] = x[0, 3] * 0.05 - 500.0
    x[0, 4, V // 2:] = 25.0                    # the maximum everywhere past the middle
    x[0, 5] = 0.0
    return x


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "fp16", "fp32"])
@pytest.mark.parametrize("vecs", [2, 31, 33, 255, 256, 257, 511, 512, 513, 1025, 4095, 4096])
def test_row_lengths_against_the_oracle(fd, orc, dtype, vecs):
    x = _rows(dtype, vecs, seed=vecs)
    rng = np.random.default_rng(vecs)
    mask = (rng.random((10, 32)) < 0.8).astype(np.uint8)
    mask[0, :6] = 1
    _, tok, _, _ = check_confidence(fd, orc, x, mask)
    assert tok[0, 2] == 0 and tok[0, 0] == 0 and tok[0, 1] == x.shape[2] - 1
    assert check_select(fd, orc, x, mask, oracle.PROFILE, 0.75) <= 2


@pytest.mark.gpu
@pytest.mark.parametrize("B, L", [(304, 32), (304, 33), (305, 1), (305, 32), (305, 70), (311, 3),
                                  (2432, 4), (2433, 4), (9729, 1)])
def test_many_rows(fd, orc, B, L):
    """The edges of how the kernels after the reduction spread rows over CTAs: up to 304 batch rows
    one to a CTA, then (L <= 32) eight, up to and beyond 304 such CTAs; 32 or (beyond 9728
    positions) more of them to a CTA."""
    w = syn.Workload("many", B, L, 1000, "bf16", 1.0, "target", 0.3, 3.0)
    x = syn.make_logits(w, seed=B + L, device="cuda")
    mask = (np.random.default_rng(B).random((B, L)) < 0.7).astype(np.uint8)
    mask[-1] = 1
    x[B // 2, 0, 999] = torch.nan
    mask[B // 2, 0] = 1
    check_confidence(fd, orc, x, mask)
    assert check_select(fd, orc, x, mask, oracle.PROFILE, 0.75) <= B // 50 + 1
    x[B // 2, 0, 999] = 1.0
    conf, tok = fd.fdllm_confidence(x, torch.from_numpy(mask).cuda())
    a, b = torch.from_numpy(mask.copy()).cuda(), torch.from_numpy(mask.copy()).cuda()
    got = fd.fdllm_select(x, a, 0.75, oracle.FACTOR)
    ref = fd.fdllm_select_from_conf(conf.nan_to_num(0.5), tok, b, 0.75, oracle.FACTOR)
    assert torch.equal(a, b) and all(torch.equal(g, r) for g, r in zip(got, ref))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "fp16", "fp32"])
def test_unusable_rows(fd, orc, dtype):
    """NaN, +inf and all -inf anywhere in a row's units make it unusable, its neighbours not."""
    x = _rows(dtype, 600, seed=3)
    V = x.shape[2]
    for l, (at, value) in enumerate([(V - 1, torch.nan), (0, torch.nan), (V // 2, torch.inf),
                                     (slice(None), -torch.inf)]):
        x[3, 2 * l, at] = value
    mask = np.ones((10, 32), np.uint8)
    check_confidence(fd, orc, x, mask)
    check_select(fd, orc, x, mask, oracle.PROFILE, 0.75)


@pytest.mark.gpu
def test_identical_rows_are_exact_ties(fd):
    """A row's result does not depend on the warp, the CTA or the mask that it is reduced in."""
    V = 8 * 1500
    row = torch.randn(V, device="cuda").to(torch.bfloat16)
    x = row.repeat(40, 32, 1).contiguous()
    for density in (1.0, 0.1):
        mask = (torch.rand((40, 32), device="cuda") < density).to(torch.uint8)
        mask[7, 7] = 1
        conf, tok = fd.fdllm_confidence(x, mask)
        on = mask != 0
        assert (conf[on] == conf[7, 7]).all() and (tok[on] == row.float().argmax()).all()


@pytest.mark.gpu
def test_scratch_of_one_partial_per_row_serves(fd, orc):
    """A workspace that holds one partial per row (what a longer vocabulary of one unit per row
    asks for) is accepted for a shorter one, under capture too."""
    x = _rows("bf16", 1025, seed=9)
    mask_np = np.ones((10, 32), np.uint8)
    need = fd.fdllm_workspace_bytes(10, 32, x.shape[2])
    small = fd.fdllm_workspace_bytes(10, 32, 8 * 8000)  # 128 KB rows: one unit each
    assert small < need
    ref = orc.select(syn.host_bits(x), mask_np, oracle.PROFILE, 0.75)
    ok = ref["margin"] >= 1e-5
    mask = torch.from_numpy(mask_np.copy()).cuda()
    ws = torch.zeros(small, dtype=torch.uint8, device="cuda")
    tok, commit, n = fd.fdllm_select_ws(x, mask, 0.75, "profile", ws)
    assert np.array_equal(n.cpu().numpy()[ok], ref["n"][ok])
    with pytest.raises(fd.FdllmError) as e:
        fd.fdllm_select_ws(x, mask, 0.75, "profile", ws[:256 + 320 * 16 - 256])
    assert e.value.status == 5
    # the library's workspace as fewer rows (no warp units) of a longer vocabulary left it, then a
    # capture
    fd.fdllm_release_workspace()
    fd.fdllm_select(torch.randn(8, 38, 8 * 8000, device="cuda").to(torch.bfloat16),
                    torch.ones((8, 38), dtype=torch.uint8, device="cuda"), 0.75)
    out = (torch.full((10, 32), -1, dtype=torch.int32, device="cuda"),
           torch.zeros((10, 32), dtype=torch.uint8, device="cuda"),
           torch.zeros((10,), dtype=torch.int32, device="cuda"))
    mask = torch.from_numpy(mask_np.copy()).cuda()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fd.fdllm_select(x, mask, 0.75, "profile", *out)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out[2].cpu().numpy()[ok], ref["n"][ok])
    assert np.array_equal(out[0].cpu().numpy()[ok], ref["tokens"][ok])


def test_static_scratch_still_holds_every_shape(cuda_lib_path):
    """What fdllm_select_static accepts: V up to 126464, any type, up to 65536 rows."""
    lib = ctypes.CDLL(cuda_lib_path)
    lib.fdllm_workspace_bytes.restype = ctypes.c_size_t
    for rows in (1, 304, 305, 4096, 65535, 65536):
        for V in range(8, 126465, 488):
            for dtype in (0, 1, 2):
                assert lib.fdllm_workspace_bytes(rows, 1, V, dtype) <= 8 << 20
