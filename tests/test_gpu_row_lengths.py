"""Steps a2-a5 and the per-rank terms at the row lengths where their kernels change size (up to
64, 128, 256, 512 and 1024 positions), on given confidences: distinct ones and few levels (long
runs of ties), against the oracle's rule and a stable sort."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

LENGTHS = [33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024]


def _rows(L, levels):
    rng = np.random.default_rng(L + levels)
    B = 6
    conf = rng.uniform(0.01, 1.0, (B, L)).astype(np.float32)
    conf[1] = 1.0 - 10.0 ** -rng.uniform(0.5, 5.0, L).astype(np.float32)  # a long prefix accepted
    if levels:
        conf = (np.ceil(conf * levels) / levels).astype(np.float32)
    mask = (rng.random((B, L)) < 0.8).astype(np.uint8)
    mask[1:3] = 1
    mask[3] = 0
    mask[4] = 0
    mask[4, L - 1] = 1
    tok = rng.integers(0, 1 << 20, (B, L)).astype(np.int32)
    return conf, mask, tok


@pytest.mark.parametrize("levels", [0, 5])
@pytest.mark.parametrize("L", LENGTHS)
def test_selection(fd, orc, L, levels):
    conf, mask, tok = _rows(L, levels)
    for mode, param in ((oracle.PROFILE, 0.75), (oracle.FACTOR, 3.0), (oracle.THRESHOLD, 0.6)):
        m = torch.from_numpy(mask.copy()).cuda()
        t, c, n = fd.fdllm_select_from_conf(torch.from_numpy(conf).cuda(),
                                            torch.from_numpy(tok).cuda(), m, param, mode)
        ref = orc.select_from_conf(conf.astype(np.float64), tok, mask, mode, param)
        ok = ref["margin"] >= 1e-12  # the rule's fixed point and the oracle's fp64 decide alike
        assert ok[[3, 4]].all()
        assert np.array_equal(n.cpu().numpy()[ok], ref["n"][ok])
        assert np.array_equal(c.cpu().numpy()[ok], ref["commit"][ok])
        assert np.array_equal(t.cpu().numpy()[ok], ref["tokens"][ok])
        assert np.array_equal(m.cpu().numpy()[ok], ref["mask"][ok])


@pytest.mark.parametrize("levels", [0, 5])
@pytest.mark.parametrize("L", [1, 2, 31, 32] + LENGTHS)
def test_terms(fd, L, levels):
    conf, mask, _ = _rows(L, levels)
    g = fd.fdllm_profile_terms(torch.from_numpy(conf).cuda(), torch.from_numpy(mask).cuda(), 0.25)
    g = {k: v.cpu().numpy() for k, v in g.items()}
    for b in range(len(conf)):
        at = np.nonzero(mask[b])[0]
        order = at[np.argsort(-conf[b, at], kind="stable")]
        m = len(order)
        assert np.array_equal(g["order"][b, :m], order) and (g["order"][b, m:] == -1).all()
        c = conf[b, order].astype(np.float64)
        n, S = np.arange(1, m + 1), np.cumsum(c)
        # two sums of up to L fp64 terms of at most 1, each within L * 2^-53 * L of the exact one
        tol = 2.0 * L * L * 2.0 ** -53
        for key, ref in (("G", np.maximum(0, S - (n - 1)) - (1 - c)), ("F", (n + 1) * c - n),
                         ("B", S - n * c), ("f_eff", 0.75 + S - n * c)):
            assert np.abs(g[key][b, :m] - ref).max(initial=0.0) <= tol
            assert np.isnan(g[key][b, m:]).all()
