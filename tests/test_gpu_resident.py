"""The resident time loop (small zones: the whole run in one launch, zda_resident.cu) against the FP64 oracle.

Shapes where its cut can go wrong: one brick and many, one to four own cells
per thread, phi cut and whole, bricks of one radius, row or z-cell, slabs that
fill a brick, no slabs, odd sizes, both r-PML forms, the axis zone, more steps
than one launch takes.  Tolerances as for every other step kernel: DFT fields
and phasors 1e-4, gradients 1e-3 (FP32 against FP64).
"""
import threading

import numpy as np
import pytest
import torch

import oracle as O
from zda_inputs import smoothed_rho, zone_tiny

pytestmark = pytest.mark.gpu

FIELD_TOL = 1e-4
GRAD_TOL = 1e-3
BASE = dict(filter_radius=0.2, beta=3.0, wavelengths=(0.9, 1.1), pulse_sigma=0.4, pulse_t0=1.6, n_steps=300)

SHAPES = {
    "tiny": dict(),
    "one_phi_cell": dict(n_phi=1, n_fold=300, r_lo=8.0),
    "two_phi_cells": dict(n_phi=2, n_fold=150, r_lo=8.0),
    "odd": dict(n_r=27, n_phi=7, n_z=45, pml_r_in=3, pml_r_out=5, pml_z=5),
    "no_slabs": dict(pml_r_in=0, pml_r_out=0, pml_z=0),
    "wide_slabs": dict(n_r=20, pml_r_in=9, pml_r_out=9, pml_z=11),
    "phi_cut": dict(n_r=16, n_phi=64, n_fold=16),
    "two_cells": dict(n_r=44, n_phi=44, n_z=50, n_fold=20),
    "three_cells": dict(n_r=50, n_phi=50, n_z=60, n_fold=20, n_steps=260),
    "four_cells": dict(n_r=60, n_phi=40, n_z=80, n_fold=20, n_steps=260),
    "long_z": dict(n_z=300, n_phi=3, n_fold=100, r_lo=6.0),
    "axis": dict(r_lo=0.0, n_fold=0, n_phi=1, pml_r_in=0, n_r=33, n_steps=500),
}


def _spec(name):
    return zone_tiny(**{**BASE, **SHAPES[name]})


def _zone(spec, form=0):
    from paper_2501_07979_gb300 import Zone
    z = Zone(spec, device=0)
    if form:
        z.set_radial_pml(form)
    return z


def _dev(x):
    return torch.tensor(np.asarray(x), dtype=torch.float32, device="cuda:0")


def _rel(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return float(np.linalg.norm((a - b).ravel()) / max(np.linalg.norm(b.ravel()), 1e-300))


def _rho(spec, seed=5):
    return smoothed_rho(spec.n_r_design, spec.n_phi, seed, mode="minmax")


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("name", list(SHAPES))
def test_resident_run_matches_oracle(name, form):
    spec = _spec(name)
    if form and spec.pml_r_in + spec.pml_r_out == 0:
        pytest.skip("the forms differ inside the r-PML only")
    rho = _rho(spec)
    z = _zone(spec, form)
    n0 = z.launches
    S = z.forward(_dev(rho))
    assert z.launches - n0 < 20                          # not a launch per step
    mon = z.monitor_dft().cpu().numpy()
    grad = z.adjoint(4.0 * S).cpu().numpy()
    I_ref, g_ref, fwd, adj = O.gradient(spec, rho, pml_form=form)
    assert _rel(S, fwd["S"]) < FIELD_TOL
    assert _rel(mon, fwd["mon"]) < FIELD_TOL
    assert _rel(np.moveaxis(z.design_dft(0).cpu().numpy(), 4, 2), fwd["des"]) < FIELD_TOL
    assert _rel(grad, g_ref) < GRAD_TOL


@pytest.mark.parametrize("name", ["tiny", "odd", "phi_cut", "two_cells", "axis"])
def test_resident_fields_match_the_split_step(name):
    """Final fields of both paths on the same density (the split step chosen explicitly)."""
    spec = _spec(name)
    a, b = _zone(spec), _zone(spec)
    b.set_kernel(0, 4, 0)
    Sa, Sb = a.forward(_dev(_rho(spec))), b.forward(_dev(_rho(spec)))
    assert _rel(Sa, Sb) < 1e-5
    assert _rel(a.fields().cpu().numpy(), b.fields().cpu().numpy()) < FIELD_TOL


def test_resident_run_longer_than_one_launch():
    spec = _spec("odd").replace(n_steps=4200)
    rho = _rho(spec)
    z = _zone(spec)
    S = z.forward(_dev(rho))
    fwd = O.forward(spec, rho)
    assert _rel(S, fwd["S"]) < FIELD_TOL
    assert _rel(z.monitor_dft().cpu().numpy(), fwd["mon"]) < FIELD_TOL


def test_resident_runs_of_two_threads_take_turns():
    """Zones of different sizes on two threads and streams: each result as if run alone, and repeatable."""
    specs = [_spec("odd"), _spec("two_cells")]
    rhos = [_dev(_rho(s)) for s in specs]
    want = [_zone(s).iteration(r) for s, r in zip(specs, rhos)]
    got = [None, None]

    def work(k):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            z = _zone(specs[k])
            got[k] = [z.iteration(rhos[k]) for _ in range(4)]

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for k in range(2):
        for I, g in got[k]:
            assert I == want[k][0] and torch.equal(g, want[k][1])


def test_resident_wait_that_runs_out_is_reported():
    from paper_2501_07979_gb300 import ZdaError
    spec = _spec("tiny")
    z = _zone(spec)
    r = _dev(_rho(spec))
    S = z.forward(r)
    z.set_wait_limit(1000, inject_timeout=True)
    with pytest.raises(ZdaError, match="ZDA_ERR_TIMEOUT"):
        z.forward(r)
    z.set_wait_limit(1 << 22)
    assert np.array_equal(z.forward(r), S)


def test_launches_of_the_split_step_stay_in_reach():
    """Event timing and the decay probe look between the launches of a step."""
    spec = _spec("tiny")
    z = _zone(spec)
    r = _dev(_rho(spec))
    S = z.forward(r)
    z.set_timing(10)
    n0 = z.launches
    S2 = z.forward(r)
    ms, n = z.timing()
    assert n > 0 and z.launches - n0 > 2 * spec.n_steps - 1 and _rel(S2, S) < 1e-5
    z.set_timing(0)
    z.set_energy_probe(20)
    S3 = z.forward(r)
    assert len(z.energy_trace()[0]) == spec.n_steps // 20 and _rel(S3, S) < 1e-5


@pytest.mark.parametrize("cell,n_r,one_launch", [(0.1, 24, True), (0.05, 24, False), (0.05, 48, True), (0.03, 64, False)])
def test_forward_runs_that_end_in_noise_keep_the_split_step(cell, n_r, one_launch):
    """zda_forward leaves the one-launch run where the final fields may have decayed: fine cells, or few
    wavelengths between the PMLs at medium ones."""
    spec = zone_tiny(dr=cell, dz=cell, n_r=n_r, n_z=48, filter_radius=1.6 * cell, beta=3.0, wavelengths=(1.0,),
                     pulse_sigma=0.4, pulse_t0=1.6, n_steps=300)
    z = _zone(spec)
    n0 = z.launches
    z.forward(_dev(_rho(spec)))
    assert (z.launches - n0 < 20) == one_launch


@pytest.mark.parametrize("n_steps", [1, 2, 4096, 4097, 4098])
def test_no_launch_of_a_single_step(n_steps):
    """A brick overwrites its state as its launch ends and its neighbours read it as theirs begin: only with two steps
    between is the second behind the first.  Runs of one step, and of one more than a launch takes, against the split
    step (FP32 rounding: 1e-5; the fields of the long runs have decayed, so their DFTs are held)."""
    spec = zone_tiny(**{**BASE, "n_steps": n_steps, "pulse_t0": 0.0})
    rho = _dev(_rho(spec))
    a, b = _zone(spec), _zone(spec)
    b.set_kernel(0, 4, 0)
    n0 = a.launches
    Sa = a.forward(rho)
    assert a.launches - n0 < 20
    Sb = b.forward(rho)
    assert _rel(Sa, Sb) < 1e-5
    if n_steps < 3:                                      # nothing has reached the monitor yet
        assert _rel(a.fields().cpu(), b.fields().cpu()) < 1e-5
    else:
        assert _rel(a.monitor_dft().cpu(), b.monitor_dft().cpu()) < 1e-5


@pytest.mark.parametrize("name", ["tiny", "two_cells"])
def test_a_run_that_gives_up_waiting_is_repeated_by_the_split_step(name):
    """One poll is less than a neighbour's packet takes: the run gives up, and the call's result is the split step's,
    bit for bit, for every entry point that may take the one-launch run."""
    spec = _spec(name)
    rho = _dev(_rho(spec))
    a, b = _zone(spec), _zone(spec)
    b.set_kernel(0, 2, 0)
    want = a.forward(rho)
    a.set_wait_limit(1)
    n0 = a.launches
    S, Sb = a.forward(rho), b.forward(rho)
    assert a.launches - n0 > 2 * spec.n_steps and np.array_equal(S, Sb)
    assert torch.equal(a.monitor_dft(), b.monitor_dft()) and torch.equal(a.fields(), b.fields())
    assert torch.equal(a.adjoint(4.0 * S), b.adjoint(4.0 * S))
    (Ia, ga), (Ib, gb) = a.iteration(rho), b.iteration(rho)
    assert Ia == Ib and torch.equal(ga, gb)
    n0 = a.launches
    assert a.time_steps(50) > 0 and a.launches - n0 >= 100
    a.set_wait_limit(1 << 22)
    n0 = a.launches
    assert np.array_equal(a.forward(rho), want) and a.launches - n0 < 20


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("name", ["tiny", "odd", "two_cells", "axis"])
def test_one_launch_errors_are_the_split_steps(name, form):
    """The coefficients of an update are rounded as often as the split step's, so the errors against 64 bits are those
    of another summation order of the same terms: within a quarter of each other."""
    spec = _spec(name)
    rho = _rho(spec)
    _, g_ref, fwd, _ = O.gradient(spec, rho, pml_form=form)
    errs = []
    for split in (False, True):
        z = _zone(spec, form)
        if split:
            z.set_kernel(0, 4, 0)
        S = z.forward(_dev(rho))
        des = np.moveaxis(z.design_dft(0).cpu().numpy(), 4, 2)
        errs.append((_rel(des, fwd["des"]), _rel(z.monitor_dft().cpu().numpy(), fwd["mon"]),
                     _rel(z.adjoint(4.0 * S).cpu().numpy(), g_ref)))
    print(name, form, errs)
    for one, split in zip(*errs):
        assert one < 1.25 * split


def test_the_default_comes_back():
    """A refused choice leaves the one-launch run, a made one ends it, and the default brings it back."""
    from paper_2501_07979_gb300 import ZdaError
    spec = _spec("tiny")
    z = _zone(spec)
    r = _dev(_rho(spec))

    def launches():
        n0 = z.launches
        z.forward(r)
        return z.launches - n0

    assert launches() < 20
    for bad in ((1, 3, 0), (3, 5, 0), (4, 4, 0), (6, 5, 0), (7, 16, 0), (0, 4, -1)):
        with pytest.raises(ZdaError, match="ZDA_ERR_ARG"):
            z.set_kernel(*bad)
    assert launches() < 20
    z.set_kernel(0, 4, 0)
    assert launches() >= 2 * spec.n_steps
    z.default_kernel()
    assert z.get_kernel() == (0, 2, 0) and launches() < 20
    z.set_kernel(2, 2, 0)
    z.set_radial_pml(1)
    z.default_kernel()
    assert launches() < 20


@pytest.mark.parametrize("name", ["tiny", "axis"])
def test_a_tuned_small_zone_keeps_its_one_launch_run(tmp_path, name):
    from paper_2501_07979_gb300.autotune import candidates, tune_zone
    spec = _spec(name)
    cache = str(tmp_path / "tiles.json")
    z = _zone(spec)
    choice, times = tune_zone(z, cache_path=cache)
    assert set(times) - set(candidates(spec)) == {(0, 2, 0)} and times[choice] == min(times.values())
    z2 = _zone(spec)
    assert tune_zone(z2, cache_path=cache) == (choice, {})
    for t in (z, z2):
        n0 = t.launches
        t.forward(_dev(_rho(spec)))
        assert choice == (0, 2, 0) and t.launches - n0 < 20


@pytest.mark.parametrize("kernel", [None, (0, 4, 0), (3, 8, 0), (4, 16, 0), (6, 16, 0)])
def test_time_steps_reports_no_timeout_of_an_earlier_owner(kernel):
    """The error word is whatever the workspace's memory held before, until a run clears it."""
    z = _zone(_spec("tiny"))
    if kernel:
        z.set_kernel(*kernel)
    z.workspace.fill_(1)                                 # (the tables are uploaded by the first run)
    assert z.time_steps(4) > 0
