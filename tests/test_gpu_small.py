"""The forms of the step that small lattices take, against the FP64 oracle: solid cells with their two
species as the pair (FP32 arithmetic, alone and in a batch, over a 16-bit reference refresh) and one
species per solid block (FP64).

Tolerances on the velocity field (relative L2): FP64 1e-11 (operation order), FP32 1e-5 (a few roundings
of 6e-8 over 40 steps), FP16 1e-2: 40 steps of a perturbed start that decays, whose stored differences are
rounded to 2^-12 of themselves, stay some ten roundings below the rest.
"""
import pytest

from klb_testutil import make_oracle, rel_l2, species_masks
from paper_2403_15768_gb300 import inputs, klb

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 1e-5, "fp16": 1e-2}
PIPE = inputs.PIPE_D3Q19_FP32.with_(name="small", ny=16, nz=16, radius=5, shell=2,
                                    couplings=(0.05, 0.02, 0.1, 0.0, 0.01))
SLAB9 = inputs.SLAB_D2Q9_FP64.with_(ny=14, width=8, shell=2)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


def _start(w):
    drho, u = inputs.perturbation(w, 6, 1e-3)
    o, lat = make_oracle(w), klb.lattice_from_workload(w)
    o.init_equilibrium(drho, u)
    lat.init_equilibrium(drho, u)
    return o, lat


def _check(o, lat, w):
    ref, (_, got) = o.observe()["u"], lat.get_field()
    for s, m in enumerate(species_masks(o.geo, w.nx)):
        assert rel_l2(got[s][:, m], ref[s][:, m]) <= TOL[w.storage], s


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("base,nx", [("pipe", 1), ("pipe", 31), ("pipe", 33), ("slab9", 32), ("slab9", 65)])
def test_small_lattices_follow_the_oracle(base, nx, storage):
    w = (PIPE if base == "pipe" else SLAB9).with_(nx=nx, storage=storage)
    o, lat = _start(w)
    o.step(40)
    lat.step(40)
    _check(o, lat, w)


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
def test_small_batch_follows_the_oracle(storage):
    ws = [PIPE.with_(nx=nx, storage=storage) for nx in (5, 40, 64)]
    pairs = [_start(w) for w in ws]
    batch = klb.Batch([lat for _, lat in pairs])
    batch.step(40)
    for (o, lat), w in zip(pairs, ws):
        o.step(40)
        _check(o, lat, w)
