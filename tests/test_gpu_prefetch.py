"""Steps that ask L2 for later rows (state buffers beyond the 129 MB L2): an x-invariant flow on a long
or wide lattice against the same cross-section with a few x planes, which asks for nothing.

The same bits are expected in every plane: each cell's arithmetic and dither depend on its row and
step alone; the 16-bit references are averages of equal values, exact over 32 and 64 of them (longer FP16
rows are compared with the oracle by the full-size tests).
"""
import numpy as np
import pytest

from paper_2403_15768_gb300 import inputs, klb

pytestmark = pytest.mark.gpu

L2_BYTES = 129e6
CASES = {
    # one chunk of 32 or 64 threads per row, several chunks with a ragged last one
    ("fp32", "narrow_blocks"): dict(nx=61, ny=140, nz=140, radius=62, shell=7),
    ("fp32", "two_warps"): dict(nx=127, ny=100, nz=100, radius=44, shell=5),
    ("fp32", "ragged_chunks"): dict(nx=1023, ny=44, nz=44, radius=18, shell=3),
    ("fp16", "narrow_blocks"): dict(nx=64, ny=200, nz=200, radius=90, shell=9),
}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


def _run(w, steps):
    lat = klb.lattice_from_workload(w)
    rng = np.random.default_rng(4)
    drho = np.repeat(1e-3 * rng.uniform(-1, 1, (3, w.nz, w.ny, 1)), w.nx, axis=3)
    u = np.repeat(1e-3 * rng.uniform(-1, 1, (3, 3, w.nz, w.ny, 1)), w.nx, axis=4)
    lat.init_equilibrium(drho, u)
    lat.step(steps)
    cells = sum(lat.species_cells(s) for s in range(3))
    return lat.get_field(), cells


@pytest.mark.parametrize("storage,case", sorted(CASES))
def test_long_lattice_equals_its_slice(storage, case):
    w = inputs.PIPE_D3Q19_FP32.with_(name="ahead", storage=storage, **CASES[storage, case])
    (d1, u1), cells = _run(w, 7)
    assert cells * 2 * 19 * (4 if storage == "fp32" else 2) > L2_BYTES
    (d2, u2), _ = _run(w.with_(nx=3 if storage == "fp32" else 32), 7)
    assert np.array_equal(d1, np.broadcast_to(d2[..., :1], d1.shape))
    assert np.array_equal(u1, np.broadcast_to(u2[..., :1], u1.shape))
