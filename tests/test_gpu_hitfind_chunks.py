"""Hit finding where its place kernel's chunks of 32 units end: planes of 31, 32,
33 and 65 one-segment wires in one call, and chunks in which more units overflow
their 128 slots than the kernel has warps (every second tick above), between
units with few or no runs.  Same bars as test_gpu_hitfind.py."""
import numpy as np
import pytest

from paper_2009_04509_gb300 import synth

from test_gpu_hitfind import check_plane, gpu_find

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dense", [(), (0, 5, 6, 7, 30, 31)])
def test_chunk_edges(dense):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_2009_04509_gb300 import build, emtk
    build.build()
    oracle.build()
    rng = np.random.default_rng(len(dense))
    planes = []
    for nwires in (31, 32, 33, 65):
        adc = rng.standard_normal((nwires, 600)).astype(np.float32)
        adc[rng.integers(0, nwires, 40), rng.integers(0, 600, 40)] = 50.0
        for w in dense:
            if w < nwires:
                adc[w, ::2] = 40.0 + rng.random(300).astype(np.float32)
                adc[w, 1::2] = 0.0
        planes.append((adc, 600, 15.0))
    ctx = emtk.emtk_create(synth.he_normal_weights(0), precision="bf16")
    try:
        for got, (adc, nticks, thr) in zip(gpu_find(emtk, ctx, planes), planes):
            check_plane(got, adc, nticks, thr)
    finally:
        emtk.emtk_destroy(ctx)
