"""The head of small launches where its hits per CTA change (one up to 256 hits, two
up to 912, four up to 2,048) and at counts that leave a CTA's last hits empty,
in an order of sums that differs from the large launches' head.  Bar: 1e-3 against
the fp64 oracle at fp32 accuracy (scores and, scaled by 1 + |z|, logits within 2e-3,
the fp32 paths' bars), and repeated calls give the same bits."""
import numpy as np
import pytest

import oracle
from paper_2009_04509_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 256, 257, 911, 913, 915, 2048, 2049])
def test_head_sizes(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_04509_gb300 import build, emtk
    build.build()
    oracle.build()
    w = synth.he_normal_weights(0, bias_std=0.1)
    x = synth.inference_patches(n, seed=n)
    xd = torch.from_numpy(x).cuda()
    ctx = emtk.emtk_create(w, precision="tf32", max_hits=2304, debug_logits=True)
    try:
        outs = [torch.full((n, 8), -1.0, device="cuda") for _ in range(2)]
        for o in outs:
            emtk.emtk_infer_patches(ctx, xd, o)
        assert emtk.emtk_check(ctx) == emtk.EMTK_OK
    finally:
        emtk.emtk_destroy(ctx)
    assert torch.equal(outs[0], outs[1])
    got = outs[0].cpu().numpy().astype(np.float64)
    logits, ref = oracle.forward(x, w)
    assert np.abs(got[:, :4] - ref).max() <= 1e-3
    assert (np.abs(got[:, 4:] - logits) / (1 + np.abs(logits))).max() <= 2e-3
