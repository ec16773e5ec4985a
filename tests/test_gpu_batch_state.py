"""State or couplings of a batch's members replaced between batch calls, at the same step: the batch goes
on from them, bit for bit as the lattice does alone."""
import numpy as np
import pytest

from paper_2403_15768_gb300 import inputs, klb

pytestmark = pytest.mark.gpu

PIPE = inputs.PIPE_D3Q19_FP32.with_(name="state", nx=19, ny=14, nz=14, radius=4, shell=2,
                                    couplings=(0.05, 0.02, 0.1, 0.0, 0.01))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


@pytest.mark.parametrize("change", ["state", "couplings"])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("before,after", [(6, 1), (7, 1), (7, 14), (33, 40), (385, 800)])
def test_member_replaced_between_batch_calls(before, after, storage, change):
    ws = [PIPE.with_(nx=nx, storage=storage) for nx in (19, 40)]
    mates, alone = ([klb.lattice_from_workload(w) for w in ws] for _ in range(2))
    for k, w in enumerate(ws):
        for lat in (mates[k], alone[k]):
            lat.init_equilibrium(*inputs.perturbation(w, k, 1e-3))
    batch = klb.Batch(mates)
    batch.step(before)
    for lat in alone:
        lat.step(before)
    for lat in (mates[1], alone[1]):
        if change == "state":
            g, u1, u2 = lat.get_state()
            lat.set_state(0.5 * g, u1, u2, before)
        else:
            lat.set_couplings(-0.01, 0.03, 0.2, 0.0, 0.05)
    batch.step(after)
    for a, b in zip(mates, alone):
        b.step(after)
        assert a.nstep == b.nstep == before + after
        for x, y in zip(a.get_state(), b.get_state()):
            assert np.array_equal(x, y)
        assert a.observables()["flow_rate"] == b.observables()["flow_rate"]
