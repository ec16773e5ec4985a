"""The step that lattices and batches of more than 4000 items run (two adjacent cells per thread, the solid rows'
species one after the other): bounce-back interfaces, phonons as waves, negative couplings, thermal noise, odd
rows, a 16-bit reference refresh, requests to L2 and the index checks of the debug build.  Each test also checks
that its sizes take this form.

Against the FP64 oracle after 4 steps of a start perturbed by 1e-3, relative L2 of each velocity field: FP32 a
few roundings of 6e-8, taken as 1e-5; 16 bits some ten roundings of 2^-12 (FP16) or 2^-9 (BF16) of a stored
difference of 3e-4 in momenta of that size: 5e-3 and 4e-2.  Thermal noise in FP32 (single-precision Box-Muller,
10 steps): 2e-4 of the largest value.
"""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

from klb_testutil import make_oracle, rel_l2, species_masks
from paper_2403_15768_gb300 import build, inputs, klb

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
L2_BYTES = 129e6
TOL = {"fp32": 1e-5, "fp16": 5e-3, "bf16": 4e-2}
NEGATIVE = (-0.02, 0.05, 0.1, 0.0, 0.01)  # negative water-electron friction
WAVES = dict(iface_bc="bounceback", phonon_wave=True, couplings=NEGATIVE)
PIPE = inputs.PIPE_D3Q19_FP32.with_(name="two_cell", ny=40, nz=40, radius=14, shell=4, couplings=(0.05, 0.02, 0.1, 0.0, 0.01))
SLAB9 = inputs.SLAB_D2Q9_FP64.with_(name="two_cell9", nx=513, ny=400, width=300, shell=50)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    klb.load_library()


def _rows(lat, w):
    return sum(lat.species_cells(s) for s in (0, 1)) // w.nx


def _takes_two_cells(lat, w):
    """Blocks of four items of 64 cells, not of species pairs (32 solid cells)."""
    batch = klb.Batch([lat])
    ok = batch.width == 128 and batch.blocks == -(-_rows(lat, w) * -(-w.nx // 64) // 4)
    batch.close()
    return ok


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("w", [PIPE.with_(nx=257), PIPE.with_(nx=257, **WAVES), PIPE.with_(nx=1023, ny=24, nz=24, radius=8, shell=3, **WAVES),
                               SLAB9.with_(**WAVES)], ids=["specular", "waves", "long_waves", "d2q9_waves"])
def test_two_cell_rows_follow_the_oracle(w, storage):
    w = w.with_(storage=storage)
    o, lat = make_oracle(w), klb.lattice_from_workload(w)
    assert _takes_two_cells(lat, w)
    drho, u = inputs.perturbation(w, 2, 1e-3)
    o.init_equilibrium(drho, u)
    lat.init_equilibrium(drho, u)
    o.step(4)
    lat.step(4)
    ref, (_, got) = o.observe()["u"], lat.get_field()
    for s, m in enumerate(species_masks(o.geo, w.nx)):
        assert rel_l2(got[s][:, m], ref[s][:, m]) <= TOL[storage], s


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx", [1, 33, 64, 191])
def test_both_forms_of_the_solid_rows_give_the_same_bits(nx, storage):
    """A lattice that alone takes species pairs, stepped in a batch that takes two cells."""
    ws = [PIPE.with_(nx=nx, ny=20, nz=20, radius=6, shell=3, storage=storage, **WAVES), PIPE.with_(nx=300, storage=storage)]
    mates, alone = [klb.lattice_from_workload(w) for w in ws], klb.lattice_from_workload(ws[0])
    assert not _takes_two_cells(alone, ws[0])
    for lat in (mates[0], alone):
        lat.init_equilibrium(*inputs.perturbation(ws[0], 3, 1e-3))
    batch = klb.Batch(mates)
    assert batch.blocks == -(-_rows(mates[0], ws[0]) * -(-nx // 64) // 4) + -(-_rows(mates[1], ws[1]) * 5 // 4)
    batch.step(70)
    alone.step(70)
    for a, b in zip(alone.get_state(), mates[0].get_state()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nx,change", [(256, {}), (257, WAVES)], ids=["specular", "waves"])
def test_noise_on_two_cells_matches_the_oracle(nx, change):
    w = PIPE.with_(nx=nx, **change)
    o, lat = make_oracle(w), klb.lattice_from_workload(w)
    assert _takes_two_cells(lat, w)
    o.init_equilibrium()
    o.set_fluctuations(1e-5, 0x5EED_1234_ABCD)
    lat.set_fluctuations(1e-5, 0x5EED_1234_ABCD)
    o.step(10)
    lat.step(10)
    f, (drho, u) = o.observe(), lat.get_field()
    for s, m in enumerate(species_masks(o.geo, w.nx)):
        ref, got = f["u"][s][:, m], u[s][:, m]
        assert np.abs(got - ref).max() <= 2e-4 * np.abs(ref).max(), s
        dr, dg = f["drho"][s][m], drho[s][m]
        assert np.abs(dg - dr).max() <= 2e-4 * max(np.abs(dr).max(), 1e-12), s


@pytest.mark.parametrize("w", [PIPE.with_(nx=128, ny=42, nz=42, radius=15), PIPE.with_(nx=101, ny=42, nz=42, radius=15, **WAVES),
                               inputs.SLAB_D2Q9_FP64.with_(nx=65, ny=60, width=40, shell=10, storage="fp32")],
                         ids=["specular", "waves", "d2q9"])
def test_noise_where_only_the_noise_free_step_takes_species_pairs(w):
    """Noise off, on and off again on lattices of up to 4000 items whose noisy steps take two cells."""
    o, lat = make_oracle(w), klb.lattice_from_workload(w)
    assert not _takes_two_cells(lat, w)
    o.init_equilibrium()
    for steps, kT in ((2, 0.0), (7, 1e-5), (3, 0.0)):
        o.set_fluctuations(kT, 99)
        lat.set_fluctuations(kT, 99)
        o.step(steps)
        lat.step(steps)
    f, (drho, u) = o.observe(), lat.get_field()
    for s, m in enumerate(species_masks(o.geo, w.nx)):
        ref, got = f["u"][s][:, m], u[s][:, m]
        assert np.abs(got - ref).max() <= 2e-4 * np.abs(ref).max(), s
        dr, dg = f["drho"][s][m], drho[s][m]
        assert np.abs(dg - dr).max() <= 2e-4 * max(np.abs(dr).max(), 1e-12), s


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_requests_to_l2_change_no_bits(storage):
    """Lattices below the 129 MB L2 that alone ask it for nothing, in a batch beyond it that does."""
    k = 1 if storage == "fp32" else 2
    ws = [PIPE.with_(nx=nx, ny=100, nz=100, radius=44, shell=5, storage=storage, **c)
          for nx, c in ((61 * k, WAVES), (48 * k, {}), (65 * k, {}))]
    mates = [klb.lattice_from_workload(w) for w in ws]
    size = [sum(lat.species_cells(s) for s in range(3)) * 2 * 19 * (4 // k) for lat in mates]
    assert max(size) < L2_BYTES < sum(size)
    alone = [klb.lattice_from_workload(w) for w in ws[:2]]
    for lat, w in zip(alone, ws):
        start = inputs.perturbation(w, 5, 1e-3)
        lat.init_equilibrium(*start)
        mates[alone.index(lat)].init_equilibrium(*start)
    klb.Batch(mates).step(35)
    for a, b in zip(alone, mates):
        a.step(35)
        for x, y in zip(a.get_state(), b.get_state()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("nx", [65, 257])
def test_non_finite_cells_are_counted(nx, storage):
    """A NaN in one electron population and an infinity in one water population (whole rows with 16-bit
    references): the species-cells counted are those whose fields are not finite."""
    w = PIPE.with_(nx=nx, storage=storage)
    o, lat = make_oracle(w), klb.lattice_from_workload(w)
    lat.step(3)
    g, u1, u2 = lat.get_state()
    masks = species_masks(o.geo, nx)
    z, y, _ = np.argwhere(masks[1])[len(np.argwhere(masks[1])) // 2]
    g[1, 5, z, y, nx - 1] = np.nan
    g[0, 3, w.nz // 2, w.ny // 2, 0] = np.inf
    lat.set_state(g, u1, u2, 3)
    drho, u = lat.get_field()
    bad = sum(int((~np.isfinite(drho[s]) | ~np.isfinite(u[s]).all(axis=0))[masks[s]].sum()) for s in range(3))
    with pytest.raises(klb.KLBError):
        lat.observables()
    assert lat.observables(allow_unstable=True)["nonfinite"] == bad > 0


CHILD = textwrap.dedent("""
    import sys
    sys.path.insert(0, {root!r})
    import torch
    from paper_2403_15768_gb300 import inputs, klb

    lib = klb.load_library()
    assert lib.klb_bounds_checked() == 1
    pipe = inputs.PIPE_D3Q19_FP32.with_(nx=257, ny=40, nz=40, radius=14, shell=4)
    wide = pipe.with_(nx=127, ny=100, nz=100, radius=44, shell=5)
    cases = [pipe, pipe.with_(storage="fp16"), pipe.with_(storage="bf16", iface_bc="bounceback"),
             pipe.with_(iface_bc="bounceback", phonon_wave=True), wide,
             inputs.SLAB_D2Q9_FP64.with_(nx=513, ny=400, width=300, shell=50, storage="fp32")]
    lats = []
    for k, w in enumerate(cases):
        lat = klb.lattice_from_workload(w)
        lat.init_equilibrium(*inputs.perturbation(w, k, 1e-3))
        lat.step(40 if lat.desc.storage > 1 else 6)
        lat.observables()
        lats.append(lat)
    klb.Batch([l for l, w in zip(lats, cases) if w.kind == 19 and w.storage == "fp32"]).step(13)
    many = [klb.lattice_from_workload(pipe.with_(nx=3, ny=10, nz=10, radius=3, shell=1)) for _ in range(60)]
    klb.Batch(many[:40]).step(7)
    klb.Batch(many[40:] + [lats[3]]).step(7)
    noisy = klb.lattice_from_workload(pipe)
    noisy.set_fluctuations(1e-5, 3)
    noisy.step(5)
    lats += [noisy] + many
    bad = [(k, l.bounds_status()) for k, l in enumerate(lats)]
    bad = [b for b in bad if b[1]]
    print("OK" if not bad else "BAD %r" % bad)
""")


def test_debug_build_has_no_out_of_range_index():
    env = dict(os.environ, KLB_LIBRARY=build.build(bounds=True))
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], env=env, capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip().splitlines()[-1] == "OK", r.stdout + r.stderr
