"""The fp32 network kernel where its split of the work changes: one hit, the
128-hit tile's edge, and launches in which a CTA has less than one tile or more
(13.8 tiles are 88 pairs per CTA on 152 SMs).  Bar: the fp32 path's,
max |score difference| <= 1e-3 against the fp64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2009_04509_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 128, 129, 1664, 1665, 1793])
def test_fp32_patches_every_split(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_04509_gb300 import build, emtk
    build.build()
    oracle.build()
    w = synth.he_normal_weights(0, bias_std=0.1)
    x = synth.inference_patches(n, seed=n)
    ctx = emtk.emtk_create(w, precision="fp32", max_hits=2048)
    try:
        scores = torch.zeros((n, 4), device="cuda")
        emtk.emtk_infer_patches(ctx, torch.from_numpy(x).cuda(), scores)
        assert emtk.emtk_check(ctx) == emtk.EMTK_OK
        got = scores.cpu().numpy().astype(np.float64)
    finally:
        emtk.emtk_destroy(ctx)
    _, ref = oracle.forward(x, w)
    assert np.abs(got - ref).max() <= 1e-3
