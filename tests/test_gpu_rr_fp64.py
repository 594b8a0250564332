"""The FP64 path's subspace diagonalisation (Cholesky of the overlap, tridiagonalisation, divide and
conquer): the blocks of wavefunctions it has to take, and each form of its launch."""
import dataclasses
import threading

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sgo():
    from paper_1603_02732_gb300 import build
    build.build()
    import paper_1603_02732_gb300 as pkg
    pkg.load_library()
    return pkg


OPTS = dict(precision="fp64", scf_tol_e=1e-10, scf_tol_rho=1e-8, max_scf=100)


# a start of small norm, and two bands that nearly agree (squared distance 8e-4, 2e-6), in every size class
@pytest.mark.parametrize("bands", [5, 40, 80, 120])
@pytest.mark.parametrize("change", ["scaled 0.03", "scaled 1e-5", "overlap 0.9996", "overlap 0.999999"])
def test_states_need_not_be_orthonormal(sgo, bands, change):
    """sgo_set_state takes wavefunctions that are not orthonormal: the evaluation from them converges to
    the same F (second order in the density error of 1e-8 per electron: below 1e-9)."""
    st = dataclasses.replace(workloads.tiny(nat=2 if bands > 5 else 1, ecut=9.0, kT=0.01), nbands=bands)
    ref = sgo.Context(st, **OPTS)
    F = ref.energy_forces()[0]
    rho, psi = ref.get_state()
    what, by = change.split()
    psi = psi.copy()
    if what == "scaled":
        psi *= float(by)
    else:
        psi[1] = float(by) * psi[0] + np.sqrt(1.0 - float(by) ** 2) * psi[1]
    ctx = sgo.Context(st, **OPTS)
    ctx.set_state(rho, psi)
    got = ctx.energy_forces()[0]  # (raises unless SGO_OK)
    assert abs(got - F) < 1e-9
    psi = ctx.get_state()[1]
    assert np.abs(psi @ psi.T - np.eye(bands)).max() < 1e-12


@pytest.mark.parametrize("missing", [0, 1, 3])
def test_nearly_as_many_bands_as_plane_waves(sgo, missing):
    """The random start is not normalised, and with (nearly) as many bands as plane waves its last
    directions are nearly dependent."""
    st = dataclasses.replace(workloads.tiny(nat=1, ecut=2.0, kT=0.01), nbands=3)
    npw = sgo.Context(st, extra_bands=0, precision="fp64").npw
    assert npw <= 128
    st = dataclasses.replace(st, nbands=npw - missing)
    ctx = sgo.Context(st, extra_bands=0, **OPTS)
    ctx.energy_forces()
    psi = ctx.get_state()[1]
    assert np.abs(psi @ psi.T - np.eye(npw - missing)).max() < 1e-11


# two sizes of one launch form, in FP64 and on the cluster of 8 CTAs
@pytest.mark.parametrize("opts,bands", [(dict(OPTS, max_scf=3), (66, 96)), (dict(OPTS, max_scf=3, rr_cluster=1), (20, 100)),
                                        (dict(precision="mixed", max_scf=3, rr_cluster=1), (20, 120))])
def test_contexts_on_two_threads(sgo, opts, bands):
    """Different contexts may be used from different threads (include/sgo.h): a small and a large
    structure evaluated side by side give what each gives alone."""
    import torch
    made = []
    for n in bands:
        st = dataclasses.replace(workloads.tiny(nat=2, ecut=9.0, kT=0.01), nbands=n)
        stream = torch.cuda.Stream()
        ctx = sgo.Context(st, stream=stream.cuda_stream, extra_bands=0, **opts)
        made.append((stream, ctx, ctx.energy_forces(check=False)[0]))
    wrong = []

    def work(ctx, want):
        for _ in range(100):
            try:
                got = ctx.energy_forces(check=False)[0]
            except Exception as e:  # noqa: BLE001
                got = str(e)
            if got != want:
                wrong.append((got, want))

    threads = [threading.Thread(target=work, args=(c, w)) for _, c, w in made]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, (len(wrong), wrong[0])


# the 2 n_b block of a Davidson step from a random start (near-dependent directions are left out of it) in
# each form of the launch on a cluster of 8 CTAs
@pytest.mark.parametrize("bands", [5, 24, 44, 60])
def test_davidson_blocks(sgo, bands):
    """Both eigensolvers converge to the same F (second order in the density error: below 1e-9)."""
    st = dataclasses.replace(workloads.tiny(nat=2 if bands > 5 else 1, ecut=9.0, kT=0.01), nbands=bands)
    F = [sgo.Context(st, extra_bands=0, eigensolver=e, **OPTS).energy_forces()[0] for e in ("cg", "davidson")]
    assert abs(F[0] - F[1]) < 1e-9


# 8, 4 and 1 CTAs per problem (9, 10 and 20 members a launch) above 64 bands, with the matrices in shared
# memory and (from about 90 bands) the factors and reflectors in global scratch
@pytest.mark.parametrize("members", [9, 10, 20])
@pytest.mark.parametrize("bands", [80, 96, 120, 128])
def test_launch_forms(sgo, members, bands):
    """A member's F and spectrum after a few iterations are bitwise those of a batch of two: the CTAs of a
    problem share its work without changing a sum."""
    st = dataclasses.replace(workloads.tiny(nat=2, ecut=9.0, kT=0.01), nbands=bands)

    def run(n):
        ctxs = [sgo.Context(st, precision="fp64", max_scf=3, autotune=0, sub_batches=1, extra_bands=0) for _ in range(n)]
        F = sgo.Batch(ctxs).energy_forces()[0]
        return F, [c.eigen()[0] for c in ctxs]

    F, eps = run(members)
    F2, eps2 = run(2)
    assert np.all(F == F2[0])
    assert all(np.array_equal(e, eps2[0]) for e in eps)


@pytest.mark.parametrize("bands", [5, 40])
def test_state_of_subnormal_overlaps(sgo, bands):
    """The reciprocals and square roots of the Cholesky cover the subnormal numbers: from wavefunctions
    scaled by 1e-156 (overlaps near 1e-312, 11 digits) the evaluation converges to the same F."""
    st = dataclasses.replace(workloads.tiny(nat=2 if bands > 5 else 1, ecut=9.0, kT=0.01), nbands=bands)
    ref = sgo.Context(st, **OPTS)
    F = ref.energy_forces()[0]
    rho, psi = ref.get_state()
    ctx = sgo.Context(st, **OPTS, extra_bands=0)
    ctx.set_state(rho, 1e-156 * psi)
    assert abs(ctx.energy_forces()[0] - F) < 1e-9
