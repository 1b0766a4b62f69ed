"""The patch gather's aligned reads at every phase of a window against its image:
hits in consecutive intervals (all phases of a 16-byte chunk, in 4- and 2-byte
elements) in the first, an inner and the last wires and intervals, in the plane's
corners and just outside it.  Bit-exact against the oracle's cut."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nwires,nticks", [(97, 6 * 101 + 5), (48, 6 * 48), (3, 6)])
@pytest.mark.parametrize("fmt", ["f32", "bf16", "fp16"])
@pytest.mark.parametrize("static", [False, True])
def test_gather_every_phase(fmt, nwires, nticks, static):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_04509_gb300 import build, emtk, synth
    build.build()
    oracle.build()
    rng = np.random.default_rng(nwires)
    ld = (nticks + 3) // 4 * 4 + 4
    adc = rng.standard_normal((nwires, ld)).astype(np.float32)
    nint = nticks // 6
    cols = sorted({b for c in (0, 24, nint // 2, nint - 24, nint - 1) for b in range(c - 2, c + 9)})
    rows = sorted({w for c in (0, 24, nwires // 2, nwires - 24, nwires - 1) for w in (c - 1, c, c + 1)})
    hits = np.array([(w, 6 * b) for w in rows for b in cols], np.int32)
    dtype = {"f32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[fmt]
    out = torch.full((len(hits), 48, 48), 7.0, device="cuda", dtype=dtype)
    a, h = torch.from_numpy(adc).cuda(), torch.from_numpy(hits).cuda()
    if static:
        emtk.emtk_extract_patches_static(a, nticks, h, out, fmt)
        torch.cuda.synchronize()
    else:
        ctx = emtk.emtk_create(synth.he_normal_weights(0), precision="bf16", max_hits=256)
        try:
            emtk.emtk_extract_patches(ctx, a, nticks, h, out, fmt)
            assert emtk.emtk_check(ctx) == emtk.EMTK_OK
        finally:
            emtk.emtk_destroy(ctx)
    want = torch.from_numpy(oracle.extract_patches(adc, nticks, hits)).to(dtype)
    assert torch.equal(out.cpu(), want)
