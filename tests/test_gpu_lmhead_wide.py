"""The LM head's wide variant (W as the M = 256 operand of a CTA pair, up to 256 or 320 rows as
its N): row counts on the edges of a group, a block and the host's choice of it, W tiles that
leave whole, split and partial last rounds over the pairs, against the oracle at the LM-head
tests' own bars."""
import numpy as np
import pytest
import torch

from gpu_util import CONF_RTOL, MARGIN, oracle_threads
from test_gpu_lmhead import bits, gemm_bound, gpu_logits, inputs

import oracle

pytestmark = pytest.mark.gpu

# (B, L, H, V, masked rows)
SHAPES = [
    (1, 3, 72, 40, 2),           # V within the even CTA's half of one tile
    (2, 20, 64, 129, 33),        # few entries in the odd CTA's half; one K-block
    (2, 40, 192, 34048, 70),     # tiles of 2 x 112 entries
    (3, 64, 72, 36480, 150),     # of 2 x 120, at the most rows that take low tiles
    (5, 32, 64, 9750, 160),      # of 2 x 96, the last one ragged
    (4, 64, 128, 300, 193),      # a group of 224: two passes over its columns
    (4, 64, 128, 300, 256),      # one group of 256: two accumulators
    (4, 65, 192, 5000, 257),     # two groups; all 20 tiles split between two pairs
    (10, 32, 256, 12000, 288),   # groups of 160 and 128; 47 tiles: no split, a round of its own
    (10, 32, 64, 25000, 288),    # the same, the last round split between the groups
    (5, 64, 128, 25000, 320),    # 98 tiles: a whole round, then a split one
    (6, 64, 136, 700, 321),      # two blocks of one group; a ragged K tail
    (9, 60, 64, 1000, 513),      # three blocks
    (14, 64, 64, 3000, 896),     # four blocks
    (16, 66, 64, 3000, 1040),    # five
    (128, 32, 64, 1500, 4096),   # sixteen: the most rows that take this variant by default
    (5, 64, 8, 20000, 320),      # H below one K-block
    (4, 64, 128, 19500, 225),    # 77 tiles: one left over, its group of 256 halved
    (4, 64, 64, 25000, 150),     # a group of 160 cut into 96 and 64
    (6, 64, 64, 19600, 384),     # two blocks of 192, one tile's two items left over
    (10, 64, 64, 6000, 600),     # three blocks of 224: too many items left over to halve
    (10, 64, 64, 3000, 577),     # halved; the last half has one row
    (13, 64, 64, 2000, 770),     # four blocks; the last half has none
]


@pytest.fixture
def wide(monkeypatch):
    monkeypatch.setenv("FDLLM_LMHEAD_GEMM", "wide")


def drawn(B, L, H, V, rows):
    h, w, mask = inputs(B, L, H, V, seed=rows)
    mask[:] = 0
    mask.reshape(-1)[np.random.default_rng(rows).permutation(B * L)[:rows]] = 1
    return h, w, mask


def check_gemm_and_reduction(fd, orc, h, w, mask, entries=None):
    """The stored accumulators (at the given vocabulary entries) within the fp32 bound of the exact
    products, and the fused confidences those of the same accumulators."""
    m = torch.from_numpy(mask).cuda()
    x = fd.fdllm_lmhead_logits(h, w, m)
    conf, tok = fd.fdllm_lmhead_confidence(h, w, m)
    assert fd.fdllm_device_status() == 0
    mk = mask.astype(bool)
    xg = x.cpu().numpy()
    at = np.arange(w.shape[0]) if entries is None else entries
    ref, mag = orc.lmhead_logits(bits(h), bits(w[torch.from_numpy(at).cuda()]), mask=mask,
                                 with_abs=True, nthreads=oracle_threads())
    err = np.abs(xg[mk][:, at].astype(np.float64) - ref[mk])
    assert (err <= gemm_bound(mag[mk], ref[mk], h.shape[-1])).all(), err.max()
    assert np.isnan(xg[~mk]).all()
    rc, rt, bad = orc.confidence(np.nan_to_num(xg, nan=0.0), mask, nthreads=oracle_threads())
    assert bad == 0
    assert np.array_equal(tok.cpu().numpy()[mk], rt[mk])
    c = conf.cpu().numpy().astype(np.float64)
    assert (np.abs(c[mk] - rc[mk]) / rc[mk]).max() <= CONF_RTOL


@pytest.mark.parametrize("B,L,H,V,rows", SHAPES)
def test_gemm_and_reduction(fd, orc, wide, B, L, H, V, rows):
    check_gemm_and_reduction(fd, orc, *drawn(B, L, H, V, rows))


# K loops longer than the ring (at most 11 stages of 64): stages reused within an item, and with two
# groups the first one held up by a full ring while the second one's accumulator is being read
LONG = [
    (10, 32, 1024, 45000, 288),  # groups of 160 and 128: two rounds of W tiles, then split ones
    (10, 32, 1024, 45000, 320),  # two groups of 160
    (10, 32, 4096, 25000, 288),  # a round, then tiles split between the groups
    (10, 32, 4096, 25000, 320),
    (8, 32, 4096, 25000, 200),   # one group, the tiles left over halved
    (9, 32, 4096, 20000, 257),   # two groups: 79 tiles
    (8, 32, 4096, 45000, 256),   # one group of 256
]


@pytest.mark.parametrize("B,L,H,V,rows", LONG)
def test_long_hidden_size(fd, orc, wide, B, L, H, V, rows):
    """Logits checked at the first and last entries and at drawn ones (every W tile among them)."""
    rng = np.random.default_rng(H + rows)
    at = np.concatenate([np.arange(300), np.arange(V - 300, V), np.arange(300, V - 300, 37),
                         rng.integers(0, V, 200)])
    check_gemm_and_reduction(fd, orc, *drawn(B, L, H, V, rows), entries=np.unique(at))


@pytest.mark.parametrize("B,L,H,V", [(48, 32, 2568, 600), (29, 53, 2568, 600),
                                     (64, 64, 2560, 300), (17, 241, 2560, 300)])
def test_either_side_of_the_choice(fd, orc, monkeypatch, B, L, H, V):
    """1536 and 1537 rows of H beyond 2560, 4096 and 4097 of H up to it, by the host's own choice."""
    monkeypatch.delenv("FDLLM_LMHEAD_GEMM", raising=False)
    monkeypatch.delenv("FDLLM_LMHEAD_BN", raising=False)
    check_gemm_and_reduction(fd, orc, *drawn(B, L, H, V, B * L - 3))


@pytest.mark.parametrize("k", [12, 26, 122])
def test_confidence_at_large_magnitude(fd, orc, wide, k):
    B, L, H, V = 9, 32, 256, 3000
    h, w, mask = inputs(B, L, H, V, seed=31 + k)
    h = h * (2.0 ** k)
    conf, tok = fd.fdllm_lmhead_confidence(h, w, torch.from_numpy(mask).cuda())
    x32 = gpu_logits(fd, h, w, mask)
    mk = mask.astype(bool)
    rc, rt, bad = orc.confidence(x32, mask, nthreads=oracle_threads())
    assert bad == 0 and np.isfinite(x32[mk]).all()
    c = conf.cpu().numpy().astype(np.float64)
    assert np.array_equal(tok.cpu().numpy()[mk], rt[mk])
    assert (np.abs(c[mk] - rc[mk]) / rc[mk]).max() <= CONF_RTOL


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_unusable_row_and_exact_ties(fd, wide, bad):
    """Identical hidden states give identical confidences in every group, block and split tile
    and under any mask; a NaN or an infinity spoils its own row alone."""
    B, L, H, V = 18, 32, 192, 25000
    h, w, _ = inputs(B, L, H, V, seed=3)
    h[:] = h[0, 0]
    h[5, 5, 17] = bad
    for share in (1.0, 0.6, 0.1):
        mask = (torch.rand((B, L), device="cuda") < share).to(torch.uint8)
        mask[5, 5] = mask[0, 0] = 1
        conf, tok = fd.fdllm_lmhead_confidence(h, w, mask)
        on = mask != 0
        on[5, 5] = False
        assert torch.isnan(conf[5, 5]) and tok[5, 5] == -1
        if share == 1.0:
            first = conf[0, 0].item()
        assert (conf[on] == first).all() and (tok[on] == tok[0, 0]).all()


def test_select_and_empty_mask(fd, orc, wide):
    B, L, H, V = 4, 100, 256, 9000
    h, w, mask = inputs(B, L, H, V, seed=5)
    x32 = gpu_logits(fd, h, w, mask)
    m = torch.from_numpy(mask.copy()).cuda()
    tok, commit, n = fd.fdllm_lmhead_select(h, w, m, 0.75)
    ref = orc.select(x32, mask, oracle.PROFILE, 0.75, nthreads=oracle_threads())
    ok = ref["margin"] >= MARGIN
    assert np.array_equal(n.cpu().numpy()[ok], ref["n"][ok])
    assert np.array_equal(tok.cpu().numpy()[ok], ref["tokens"][ok])
    assert np.array_equal(m.cpu().numpy()[ok], ref["mask"][ok])
    m.zero_()
    tok, commit, n = fd.fdllm_lmhead_select(h, w, m, 0.75)
    assert (n == 0).all() and (commit == 0).all() and fd.fdllm_device_status() == 0


def test_capture_with_a_smaller_workspace(fd, monkeypatch):
    """Under capture, a workspace that holds only the tile variants' partials still serves."""
    monkeypatch.delenv("FDLLM_LMHEAD_GEMM", raising=False)
    B, L, H, V = 28, 32, 64, 60000
    h, w, mask = inputs(B, L, H, V, seed=9)
    m = torch.from_numpy(mask).cuda()
    conf, tok = fd.fdllm_lmhead_confidence(h, w, m)
    fd.fdllm_release_workspace()
    # more rows of a shorter vocabulary: room for this call's tile partials, not for the wide ones
    big = torch.randn(33, 32, H, device="cuda").to(torch.bfloat16)
    fd.fdllm_lmhead_confidence(big, w[:36000],
                               torch.ones((33, 32), dtype=torch.uint8, device="cuda"))
    c2, t2 = torch.zeros_like(conf), torch.zeros_like(tok)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fd.fdllm_lmhead_confidence(h, w, m, c2, t2)
    g.replay()
    torch.cuda.synchronize()
    on = m != 0
    assert torch.equal(tok[on], t2[on])
    assert ((conf[on] - c2[on]).abs() / conf[on]).max() <= 2 * CONF_RTOL
