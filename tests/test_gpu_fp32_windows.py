"""The fp32 network kernel's own window read: every phase of a window against the
image's 16-byte chunks, windows that reach into the zero border, hits outside the
plane, duplicates, a ragged plane, and several chunks of max_hits.  Reading the
windows and reading the same patches cut before must give the same bits, because
the two calls split the work alike."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_hits", [4096, 96])
def test_windows_equal_patches(max_hits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_04509_gb300 import build, emtk, synth
    build.build()
    rng = np.random.default_rng(3)
    nwires, nticks = 61, 6 * 83 + 5
    adc = torch.from_numpy(rng.normal(0, 20, (nwires, 504)).astype(np.float32)).cuda()
    hits = [(w, 6 * b + 1) for w in (0, 1, 23, 30, 59, 60) for b in list(range(0, 10)) + list(range(36, 50)) + [82, 83]]
    hits += [(-1, 60), (61, 60), (30, -7), (30, 6 * 140), (-400, 5), (2000, 90000), (30, 241), (30, 241)]
    h = torch.tensor(hits, dtype=torch.int32, device="cuda")
    n = len(hits)
    w = synth.he_normal_weights(0, bias_std=0.1)
    ctx = emtk.emtk_create(w, precision="fp32", max_hits=max_hits, debug_logits=True)
    try:
        got, want = (torch.full((n, 8), -1.0, device="cuda") for _ in range(2))
        patches = torch.empty(n, 48, 48, device="cuda")
        emtk.emtk_infer(ctx, adc, nticks, h, got)
        emtk.emtk_extract_patches(ctx, adc, nticks, h, patches, "f32")
        emtk.emtk_infer_patches(ctx, patches, want)
        assert emtk.emtk_check(ctx) == emtk.EMTK_OK
    finally:
        emtk.emtk_destroy(ctx)
    assert torch.equal(got, want)
    assert torch.equal(got[-1], got[-2])
