"""The patch cut of a plane whose interval image has more than 2^31 column pairs
(90 million wires of 6 ticks: 2.9 GB of samples), where the image kernel counts
pairs in 64 bits: patches at the plane's first, inner and last wires, bit-exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_more_than_2_31_pairs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB of free device memory")
    from paper_2009_04509_gb300 import build, emtk, synth
    build.build()
    nwires = 90_000_000
    adc = torch.zeros(nwires, 8, device="cuda")
    adc[:, 2] = torch.arange(nwires, device="cuda") % 251 * 6.0  # interval value: wire % 251
    wires = [0, 30, 76_695_844, 76_695_850, nwires // 2, nwires - 1]  # 2^31 pairs end near wire 76,695,820
    hits = torch.tensor([[w, 0] for w in wires], dtype=torch.int32, device="cuda")
    out = torch.full((len(wires), 48, 48), -1.0, device="cuda", dtype=torch.bfloat16)
    ctx = emtk.emtk_create(synth.he_normal_weights(0), precision="bf16", max_hits=256)
    try:
        emtk.emtk_extract_patches(ctx, adc, 6, hits, out, "bf16")
        assert emtk.emtk_check(ctx) == emtk.EMTK_OK
    finally:
        emtk.emtk_destroy(ctx)
    want = np.zeros((len(wires), 48, 48), np.float32)
    for k, w in enumerate(wires):
        for r in range(48):
            x = w - 24 + r
            if 0 <= x < nwires:
                want[k, r, 24] = x % 251
    assert torch.equal(out.float().cpu(), torch.from_numpy(want))
