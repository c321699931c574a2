"""Batched NLS at the sizes where the launch splits the work differently: the
group-tile pass's tile width and span, and the right-hand sides a warp grabs at
once, follow the number of right-hand sides. Every split does the same
arithmetic per right-hand side, so a batch must give the bits its parts give.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nmf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1509_09313_gb300 as lib
    return lib


# One tile per SM (64 x 152 right-hand sides) and its neighbours, a tile's
# edges, spans of several tiles, grabs of one to eight.
@pytest.mark.parametrize("nrhs", [1, 31, 33, 65, 9727, 9728, 9729, 40000, 170001])
@pytest.mark.parametrize("k,warm", [(10, False), (10, True), (50, False), (100, True)])
def test_bpp_batch_equals_its_parts(nmf, nrhs, k, warm):
    G, _ = synth.nls_batch(k, 1, seed=40 + k)
    rng = np.random.default_rng(nrhs + k)
    # Two thirds of the right-hand sides have positive solutions (the
    # all-passive group), the others mixed signs.
    X = rng.uniform(0.1, 1.0, (nrhs, k)) - (rng.random((nrhs, k)) < 0.2) * (np.arange(nrhs) % 3 == 0)[:, None]
    B = torch.from_numpy((X @ G).astype(np.float32)).cuda()
    Gd = torch.from_numpy(G).cuda()
    pin = nmf.bool_to_passive(torch.from_numpy(X > 0)).cuda() if warm else None
    group = 1   # the SIMT pass: the bits of the per-warp solves
    old = nmf.nmf_nls_bpp_get_shape(k)
    nmf.nmf_nls_bpp_set_shape(k, 8, 8, group)
    try:
        whole = nmf.nmf_nls_bpp(Gd, B, pin)
        cuts = sorted({0, min(nrhs, 500), nrhs // 3, nrhs})
        for a, b in zip(cuts[:-1], cuts[1:]):
            part = nmf.nmf_nls_bpp(Gd, B[a:b].contiguous(),
                                   None if pin is None else pin[a:b].contiguous())
            for name in ("X", "passive", "rounds", "status"):
                assert torch.equal(part[name], whole[name][a:b]), (name, a, b)
    finally:
        nmf.nmf_nls_bpp_set_shape(k, *old)
