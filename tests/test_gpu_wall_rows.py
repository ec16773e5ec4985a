"""Rows at walls and interfaces of the two-cell step: x-moving populations that bounce back (both
columns selected at run time) and several faces per cell, at the ends of rows and chunks, against the
FP64 oracle.

Tolerances on the velocity field (relative L2) after 4 steps of a start perturbed by 1e-3.  FP32: a
few roundings of 6e-8, taken as 1e-5.  16 bits: a stored difference of about 3e-4 is rounded to
2^-12 (FP16) or 2^-9 (BF16) of itself, 19 populations and 4 steps add up to some ten of these in a
momentum of some 3e-4: 5e-3 and 4e-2.  A wrong column on a tenth of the rows would show as some 0.3.
"""
import numpy as np
import pytest

from klb_testutil import make_oracle, rel_l2, species_masks
from paper_2403_15768_gb300 import inputs, klb

pytestmark = pytest.mark.gpu

BASE = inputs.PIPE_D3Q19_FP32.with_(name="wall_rows", ny=20, nz=20, radius=6, shell=2,
                                    couplings=(0.05, 0.02, 0.1, 0.0, 0.01))
TOL = {"fp32": 1e-5, "fp16": 5e-3, "bf16": 4e-2}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("iface", ["specular", "bounceback"])
@pytest.mark.parametrize("nx", [1, 2, 33, 257])
def test_wall_rows_follow_the_oracle(nx, iface, storage):
    w = BASE.with_(nx=nx, iface_bc=iface, storage=storage)
    drho, u = inputs.perturbation(w, 2, 1e-3)
    o, lat = make_oracle(w), klb.lattice_from_workload(w)
    o.init_equilibrium(drho, u)
    lat.init_equilibrium(drho, u)
    o.step(4)
    lat.step(4)
    ref, (_, got) = o.observe()["u"], lat.get_field()
    for s, m in enumerate(species_masks(o.geo, w.nx)):
        assert rel_l2(got[s][:, m], ref[s][:, m]) <= TOL[storage], s
    assert np.isfinite(lat.observables()["flow_rate"])
