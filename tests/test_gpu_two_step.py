"""The two-steps-per-launch form (zda_two.cu) against the FP64 oracle and the split step.

Shapes where its tiles can go wrong: wedges that a tile holds whole and wedges
cut in phi (with a ragged last tile), one phi cell, radius ranges of a few
radii, slabs that fill a range, no slabs, even and odd step counts (the last
odd step is a split step on the buffer it finds).  Tolerances as for every
other step kernel: DFT fields and phasors 1e-4, gradients 1e-3.
"""
import numpy as np
import pytest
import torch

import oracle as O
from zda_inputs import rho_for, smoothed_rho, zone_cfg2, zone_patch, zone_tiny

pytestmark = pytest.mark.gpu

FIELD_TOL = 1e-4
GRAD_TOL = 1e-3
BASE = dict(filter_radius=0.2, beta=3.0, wavelengths=(0.85, 1.0, 1.2), pulse_sigma=0.4, pulse_t0=1.6, n_steps=300)
SHAPES = {
    "tiny": dict(),
    "odd_steps": dict(n_steps=301),
    "one_phi_cell": dict(n_phi=1, n_fold=300, r_lo=8.0),
    "whole_wedge": dict(n_phi=20, n_fold=30, n_z=46, n_r=27, pml_r_in=3, pml_r_out=5),
    "cut_wedge": dict(n_phi=37, n_fold=24, n_steps=301),
    "wide_slabs": dict(n_r=20, pml_r_in=9, pml_r_out=9, pml_z=12, n_phi=33, n_fold=24),
    "no_slabs": dict(pml_r_in=0, pml_r_out=0, pml_z=0),
    "long_z": dict(n_z=150, n_phi=9, n_fold=40),
}
KERNELS = [(16, 0), (8, 0), (16, 5), (4, 3)]


def _spec(name):
    return zone_tiny(**{**BASE, **SHAPES[name]})


def _dev(x):
    return torch.tensor(np.asarray(x), dtype=torch.float32, device="cuda:0")


def _rel(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return float(np.linalg.norm((a - b).ravel()) / max(np.linalg.norm(b.ravel()), 1e-300))


def _zone(spec, *kernel):
    from paper_2501_07979_gb300 import Zone
    z = Zone(spec, device=0)
    if kernel:
        z.set_kernel(*kernel)
    return z


@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("name", list(SHAPES))
def test_two_step_run_matches_oracle(name, kernel):
    spec = _spec(name)
    rho = smoothed_rho(spec.n_r_design, spec.n_phi, 5, mode="minmax")
    z = _zone(spec, 6, *kernel)
    S = z.forward(_dev(rho))
    mon, des = z.monitor_dft().cpu().numpy(), np.moveaxis(z.design_dft(0).cpu().numpy(), 4, 2)
    grad = z.adjoint(4.0 * S).cpu().numpy()
    _, g_ref, fwd, _ = O.gradient(spec, rho)
    assert _rel(S, fwd["S"]) < FIELD_TOL
    assert _rel(mon, fwd["mon"]) < FIELD_TOL
    assert _rel(des, fwd["des"]) < FIELD_TOL
    assert _rel(grad, g_ref) < GRAD_TOL


@pytest.mark.parametrize("name", list(SHAPES))
def test_two_step_fields_match_the_split_step(name):
    spec = _spec(name)
    rho = _dev(smoothed_rho(spec.n_r_design, spec.n_phi, 6, mode="minmax"))
    a, b = _zone(spec, 6, 16, 0), _zone(spec, 0, 4, 0)
    Sa, Sb = a.forward(rho), b.forward(rho)
    assert _rel(Sa, Sb) < 1e-5
    assert _rel(a.fields().cpu().numpy(), b.fields().cpu().numpy()) < FIELD_TOL


def test_two_step_default_large_zone_and_its_fallbacks():
    """A zone of the default rule's size: same results as the split step, also under the event timing and the
    decay probe (which takes split steps)."""
    spec = zone_patch(200.0, 40)
    rho = _dev(smoothed_rho(spec.n_r_design, spec.n_phi, 7, mode="minmax"))
    z, ref = _zone(spec), _zone(spec, 0, 16, 0)
    assert z.get_kernel()[0] == 6
    want, S = ref.forward(rho), z.forward(rho)
    assert _rel(S, want) < 1e-5
    assert _rel(z.fields().cpu().numpy(), ref.fields().cpu().numpy()) < FIELD_TOL
    z.set_timing(8)
    assert np.array_equal(z.forward(rho), S)
    ms, n = z.timing()
    assert n == 5 and ms[0] > 0
    z.set_timing(0)
    z.set_energy_probe(10)
    assert _rel(z.forward(rho), S) < 1e-5 and len(z.energy_trace()[0]) == 4
    z.set_energy_probe(0)
    assert np.array_equal(z.forward(rho), S)
    z.set_radial_pml(1)
    assert z.get_kernel()[0] == 0


def test_two_step_refuses_what_it_does_not_implement():
    from paper_2501_07979_gb300 import ZdaError
    for spec, form in ((_spec("tiny").replace(n_z=41), 0), (_spec("tiny").replace(pml_z=5), 0), (_spec("tiny"), 1)):
        z = _zone(spec)
        if form:
            z.set_radial_pml(1)
        with pytest.raises(ZdaError, match="ZDA_ERR_ARG"):
            z.set_kernel(6, 16, 0)


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("kernel", [(6, 16, 0), (3, 8, 0), (1, 2, 0)])
def test_final_fields_of_a_replayed_lens_run(kernel, use_graph):
    """An odd number of launches leaves the fields in the second buffer, also where the run was a replayed graph and
    another run of the zone came in between; and a kernel chosen after a run does not move them."""
    from paper_2501_07979_gb300.lens import Lens
    spec = _spec("tiny").replace(n_steps=302 if kernel[0] == 6 else 301)
    rho = _dev(smoothed_rho(spec.n_r_design, spec.n_phi, 8, mode="minmax"))
    z = _zone(spec, *kernel)
    lens = Lens([z], use_graph=use_graph)
    lens.forward([rho])
    want = z.fields().clone()
    z.time_steps(40)
    lens.forward([rho])
    assert torch.equal(torch.view_as_real(z.fields()), torch.view_as_real(want))
    z.set_kernel(0, 4, 0)
    assert torch.equal(torch.view_as_real(z.fields()), torch.view_as_real(want))


def test_final_fields_outlive_a_change_of_the_radial_pml():
    spec = zone_patch(200.0, 38)
    z = _zone(spec)
    z.forward(_dev(smoothed_rho(spec.n_r_design, spec.n_phi, 9, mode="minmax")))
    want = z.fields().clone()
    z.set_radial_pml(1)
    assert torch.equal(torch.view_as_real(z.fields()), torch.view_as_real(want))


@pytest.mark.parametrize("use_graph", [True, False])
def test_a_timeout_under_the_decay_probe_is_reported_by_the_lens(use_graph):
    """Under the decay probe a large default zone runs its E updates on TMA tiles, whose waits are bounded: the lens
    reads their error word, in the captured run and in a replayed one, and not that of a run without the probe."""
    from paper_2501_07979_gb300 import ZdaError
    from paper_2501_07979_gb300.lens import Lens
    spec = zone_cfg2(n_steps=300)
    rho = _dev(rho_for(spec, 2))
    z = _zone(spec)
    assert z.get_kernel()[0] == 6
    lens = Lens([z], use_graph=use_graph)
    z.set_energy_probe(50)
    z.set_wait_limit(1000, inject_timeout=True)
    for _ in range(2):
        with pytest.raises(ZdaError, match="ZDA_ERR_TIMEOUT"):
            lens.forward([rho])
    z.set_energy_probe(0)
    S = lens.forward([rho])                              # two-step launches: nothing waits
    z.set_energy_probe(50)
    z.set_wait_limit(1 << 22)
    assert _rel(lens.forward([rho]), S) < 1e-5


@pytest.mark.parametrize("name", ["cut_wedge", "whole_wedge", "wide_slabs", "no_slabs"])
def test_two_step_errors_are_the_split_steps(name):
    """An update adds its curl to the field in one rounding, as in the split step, so the errors against 64 bits are
    those of another summation order of the same terms: within a quarter of each other."""
    spec = _spec(name)
    rho = smoothed_rho(spec.n_r_design, spec.n_phi, 5, mode="minmax")
    _, g_ref, fwd, _ = O.gradient(spec, rho)
    errs = []
    for kernel in ((6, 16, 0), (0, 4, 0)):
        z = _zone(spec, *kernel)
        S = z.forward(_dev(rho))
        des = np.moveaxis(z.design_dft(0).cpu().numpy(), 4, 2)
        errs.append((_rel(des, fwd["des"]), _rel(z.monitor_dft().cpu().numpy(), fwd["mon"]),
                     _rel(z.adjoint(4.0 * S).cpu().numpy(), g_ref)))
    print(name, errs)
    for two, split in zip(*errs):
        assert two < 1.25 * split
