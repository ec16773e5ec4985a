"""The observation pass (FP32 arithmetic) against sums of the downloaded fields: fewer items than one
block, ragged 64-cell segments, and more items than the resident grid takes in one turn.

get_field computes each cell with the one-cell arithmetic, the pass with the two-cell one: FP32
roundings of 6e-8 of velocities of some 2e-3 apart, so sums agree to 1e-6 of the sum of magnitudes and
the largest change to 1e-9.
"""
import numpy as np
import pytest

from klb_testutil import oracle_geometry, species_masks
from paper_2403_15768_gb300 import inputs, klb

pytestmark = pytest.mark.gpu

BASE = inputs.PIPE_D3Q19_FP32.with_(name="observe", couplings=(0.05, 0.02, 0.1, 0.0, 0.01))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("size", [dict(nx=1, ny=10, nz=10, radius=3, shell=1),
                                  dict(nx=65, ny=24, nz=24, radius=8, shell=3),
                                  dict(nx=195, ny=56, nz=56, radius=24, shell=3)])
def test_observables_are_sums_of_the_fields(size, storage):
    w = BASE.with_(storage=storage, **size)
    lat = klb.lattice_from_workload(w)
    drho, u = inputs.perturbation(w, 3, 1e-3)
    lat.init_equilibrium(drho + 5e-4, u + 1e-3)
    lat.step(5)
    _, u_prev = lat.get_field()
    lat.step(1)
    obs = [lat.observables() for _ in range(2)]
    assert repr(obs[0]) == repr(obs[1])  # the block count starts from 0 again (NaN fits compare too)
    d, u = lat.get_field()
    m = species_masks(oracle_geometry(w), w.nx)
    ux = [u[s, 0][m[s]] for s in range(3)]
    size_of = [np.abs(v).sum() for v in ux]
    assert abs(obs[0]["flow_rate"] - ux[0].sum() / w.nx) <= 1e-6 * size_of[0] / w.nx
    for s in range(3):
        assert abs(obs[0]["mean_u"][s] - ux[s].mean()) <= 1e-6 * size_of[s] / len(ux[s])
        assert abs(obs[0]["momentum"][s] - ((1 + d[s][m[s]]) * ux[s]).sum()) <= 1e-6 * size_of[s]
        assert abs(obs[0]["mass"][s] - d[s][m[s]].sum()) <= 1e-6 * np.abs(d[s][m[s]]).sum()
    change = max(np.abs(ux[s] - u_prev[s, 0][m[s]]).max() for s in range(3))
    assert abs(obs[0]["residual"] - change) <= 1e-9
    assert obs[0]["nonfinite"] == 0 and obs[0]["clipped"] == 0
