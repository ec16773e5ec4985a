"""Batches of more members than one launch's parameters hold and too few cells for several launches (one
launch over the device copies of the argument records): species pairs and cell pairs of the solid rows,
one-warp and four-warp blocks, FP64 with and without the species split, over a 16-bit reference refresh.
Bit-identical to stepping alone."""
import numpy as np
import pytest

from paper_2403_15768_gb300 import inputs, klb

pytestmark = pytest.mark.gpu

PIPE = inputs.PIPE_D3Q19_FP32.with_(name="table", ny=10, nz=10, radius=3, shell=1,
                                    couplings=(0.05, 0.02, 0.1, 0.0, 0.01))
SLAB9 = inputs.SLAB_D2Q9_FP64.with_(name="table9", ny=20, width=14, shell=3)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("base,nx,n", [(PIPE, 3, 40), (PIPE, 70, 90), (SLAB9, 33, 37), (SLAB9, 64, 300)],
                         ids=["pipe-40", "pipe-90", "slab9-37", "slab9-300"])
def test_table_launch_matches_stepping_alone(base, nx, n, storage):
    ws = [base.with_(nx=nx + k % 3, storage=storage) for k in range(n)]
    mates = [klb.lattice_from_workload(w) for w in ws]
    pick = sorted({0, 1, 35, 36, n // 2, n - 1})
    alone = {k: klb.lattice_from_workload(ws[k]) for k in pick}
    for k in pick:
        start = inputs.perturbation(ws[k], k, 1e-3)
        mates[k].init_equilibrium(*start)
        alone[k].init_equilibrium(*start)
    batch = klb.Batch(mates)
    batch.step(39)
    batch.autotune(2)
    batch.step(31)
    for k in pick:
        alone[k].step(39 + 9 + 31)
        for a, b in zip(alone[k].get_state(), mates[k].get_state()):
            assert np.array_equal(a, b), k


@pytest.mark.parametrize("n", [3, 25, 26])
def test_fp64_batch_form_matches_stepping_alone(n):
    """FP64 slabs of 96 warps that alone keep one species per solid block: in a batch as long as all its
    warps fit the chip (25 members), both species per block beyond."""
    w = SLAB9.with_(nx=64, ny=40, width=32, shell=4, storage="fp64")
    mates, alone = [klb.lattice_from_workload(w) for _ in range(n)], klb.lattice_from_workload(w)
    for lat in (mates[0], mates[-1], alone):
        lat.init_equilibrium(*inputs.perturbation(w, 4, 1e-3))
    batch = klb.Batch(mates)
    assert (batch.blocks == n * (32 + 16) * 2) == (n <= 25)
    batch.step(25)
    alone.step(25)
    for lat in (mates[0], mates[-1]):
        for a, b in zip(alone.get_state(), lat.get_state()):
            assert np.array_equal(a, b)
