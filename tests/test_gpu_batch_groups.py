"""Batches of more lattices than one launch's parameters hold: bit-identical to stepping alone, in
several launches per step (many blocks) and in one launch over the device table (few)."""
import numpy as np
import pytest

from paper_2403_15768_gb300 import inputs, klb

pytestmark = pytest.mark.gpu

PIPE = inputs.PIPE_D3Q19_FP32.with_(name="group", shell=2, couplings=(0.05, 0.02, 0.1, 0.0, 0.01))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("n,side,nx", [(36, 14, 3), (37, 14, 3), (57, 14, 3), (37, 44, 130), (113, 30, 5)])
def test_many_members_match_stepping_alone(n, side, nx, storage):
    ws = [PIPE.with_(nx=nx + k % 3, ny=side, nz=side, radius=side // 2 - 2 - k % 2, storage=storage) for k in range(n)]
    lats = [klb.lattice_from_workload(w) for w in ws]
    pick = sorted({0, 1, 35, min(36, n - 1), n // 2, n - 1})
    alone = {k: klb.lattice_from_workload(ws[k]) for k in pick}
    for k in pick:
        start = inputs.perturbation(ws[k], k, 1e-3)
        lats[k].init_equilibrium(*start)
        alone[k].init_equilibrium(*start)
    batch = klb.Batch(lats)
    batch.step(39)
    for k in pick:
        alone[k].step(39)
        for a, b in zip(lats[k].get_state(), alone[k].get_state()):
            assert np.array_equal(a, b), k
