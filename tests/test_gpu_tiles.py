"""GPU kernels at the sizes where their work split can go wrong: tile and block edges,
remainders, the smallest and largest of a range.  Each against plain NumPy in FP64."""
import dataclasses

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


def _with_bands(st, nbands):
    return dataclasses.replace(st, nbands=nbands)


# carried bands: exactly one and just over one tile group, block of 16 groups, two blocks;
# plane waves below 4096, between, and above 8192 (the K chunk and row rules)
@pytest.mark.parametrize("name,bands", [("tiny", 5), ("tiny", 12), ("tiny", 13), ("tiny", 60), ("tiny", 59),
                                        ("tiny", 63), ("tiny", 121), ("de", 81), ("layer", 49)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("mixed", 2e-6)])
def test_subspace_products_at_tile_edges(sgo, name, bands, precision, tol):
    """X^T Y, X^T X (mirrored tiles) and Y <- alpha M^T X + beta Y on the CUDA-core products,
    relative to the sums of magnitudes: K eps for a sum of K terms is 1e-12 in FP64 at the
    largest K here and its statistical growth sqrt(K) eps 2e-14; FP32 chunks 2e-6."""
    base = dict(tiny=workloads.tiny(nat=2, ecut=6.0), de=workloads.de_candidate(44), layer=workloads.honeycomb24())[name]
    ctx = sgo.Context(_with_bands(base, bands), precision=precision, gemm_tc=0)
    rng = np.random.default_rng(31)
    x, y = rng.normal(size=(2, bands, ctx.npw))
    norm = np.sqrt((x ** 2).sum(1))[:, None] * np.sqrt((y ** 2).sum(1))[None, :]
    assert np.abs(ctx.subspace_matrix(x, y) - x @ y.T).max() <= tol * norm.max()
    m = rng.normal(size=(bands, bands))
    out = ctx.block_update(x, m, -1.5, 0.5, y)
    ref = -1.5 * (m.T @ x) + 0.5 * y
    assert (np.abs(out - ref) / (1.5 * (np.abs(m).T @ np.abs(x)) + 0.5 * np.abs(y))).max() <= tol


# the tensor-core rotation: one tile of plane waves and many, output bands on either side of the 16s and
# 32s of the matrix image, the largest
@pytest.mark.parametrize("name,bands", [("tiny", 5), ("tiny", 16), ("tiny", 17), ("tiny", 33), ("tiny", 124), ("de", 81), ("layer", 49)])
def test_block_update_tensor_cores(sgo, name, bands):
    """Y <- alpha M^T X + beta Y in 3xTF32, relative to the sums of magnitudes: the split keeps 21 bits of
    each factor and drops lo lo, 4e-7, and FP32 sums of up to 124 terms add 1e-6 at most."""
    base = dict(tiny=workloads.tiny(nat=2, ecut=6.0), de=workloads.de_candidate(44), layer=workloads.honeycomb24())[name]
    ctx = sgo.Context(_with_bands(base, bands), precision="mixed")
    rng = np.random.default_rng(32)
    x, y = rng.normal(size=(2, bands, ctx.npw))
    m = rng.normal(size=(bands, bands))
    out = ctx.block_update(x, m, -1.5, 0.5, y)
    ref = -1.5 * (m.T @ x) + 0.5 * y
    assert (np.abs(out - ref) / (1.5 * (np.abs(m).T @ np.abs(x)) + 0.5 * np.abs(y))).max() <= 2e-6


# carried bands (requested + 4 + requested / 32): one leaf and two of the divide and conquer, the
# edges of every size class, the largest subspace of one CTA, and beyond it in FP64
@pytest.mark.parametrize("carried", [9, 16, 17, 32, 33, 64, 65, 96, 97, 128, 129, 184])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_subspace_eigensolve_sizes(sgo, carried, precision):
    """The one-CTA eigensolve against the cluster's (rr_cluster = 1) on the same structure: F, the
    occupied eigenvalues and the orthonormality of the bands.  Both stop at the same rule: F is
    second order in the density error (1e-8 per electron in FP64: below 1e-10; 1e-6 mixed, plus
    FP32 sums: 2e-6), an eigenvalue first order; the bands are orthonormal to n eps of the last
    rotation's precision (3xTF32 on the mixed path)."""
    bands = next(b for b in range(1, carried) if b + 4 + b // 32 == carried)
    st = _with_bands(workloads.tiny(nat=2 if bands < 12 else 3, ecut=9.0, kT=0.01), bands) if bands >= 9 else \
        _with_bands(workloads.tiny(nat=1, ecut=9.0, kT=0.01), bands)
    tol = dict(scf_tol_e=1e-10, scf_tol_rho=1e-8) if precision == "fp64" else dict(scf_tol_e=1e-7, scf_tol_rho=1e-6)
    res = []
    for cluster in (-1, 1):
        ctx = sgo.Context(st, precision=precision, rr_cluster=cluster, max_scf=100, **tol)
        # (mixed: 1e-6 is the FP32 floor of the density residual; the status is not asserted)
        F, _ = ctx.energy_forces(check=precision == "fp64")
        res.append((F, *ctx.eigen()))
        psi = ctx.get_state()[1]
        assert np.abs(psi @ psi.T - np.eye(bands)).max() < (1e-12 if precision == "fp64" else 2e-5)
        assert ctx.stats()["jacobi_cap_hits"] == 0
    occ = res[0][2] > 1e-6
    assert abs(res[0][0] - res[1][0]) < (1e-9 if precision == "fp64" else 4e-6)
    assert np.abs(res[0][1] - res[1][1])[occ].max() < (1e-7 if precision == "fp64" else 1e-4)


# plane lengths: smallest, one plane and several per CTA, odd, the largest; fewer z-planes than a
# block; band counts below, at and above the cluster's CTAs
@pytest.mark.parametrize("grid,bands,ecut", [((10, 10, 10), 5, 0.5), ((12, 16, 10), 3, 0.6), ((25, 27, 12), 16, 1.0),
                                             ((45, 25, 16), 17, 1.0), ((72, 72, 10), 18, 0.6), ((64, 10, 15), 31, 0.9)])
def test_density_sizes_mixed(sgo, grid, bands, ecut):
    """rho(r) = (1/Omega) sum_n occ_n |psi_n(r)|^2 from NumPy's FP64 transform, for FP32 bands with
    some occupations zero: 2e-6 of the largest value (the FP32 line transforms' 1e-7 a value, log N
    stages, squared)."""
    st = dataclasses.replace(workloads.tiny(nat=1, ecut=ecut, kT=0.0, nbands=bands), fft=grid)
    st = dataclasses.replace(st, cell=np.diag([10.0, 11.0, 12.0]), pos=np.array([[1.0, 2.0, 3.0]]))
    ctx = sgo.Context(st, precision="mixed", extra_bands=0)
    rng = np.random.default_rng(4)
    psi = rng.normal(size=(bands, ctx.npw)).astype(np.float32).astype(np.float64)
    occ = np.where(np.arange(bands) % 5 == 3, 0.0, rng.uniform(0.0, 2.0, size=bands))
    m = ctx.basis()[1:]
    rho = np.zeros(grid)
    for n in range(bands):
        box = np.zeros(grid, complex)
        c = (psi[n, 1::2] + 1j * psi[n, 2::2]) / np.sqrt(2.0)
        box[tuple(m.T % np.array(grid)[:, None])] = c
        box[tuple(-m.T % np.array(grid)[:, None])] = c.conj()
        box[0, 0, 0] = psi[n, 0]
        rho += occ[n] * np.abs(np.fft.ifftn(box) * box.size) ** 2
    rho /= abs(np.linalg.det(st.cell))
    got = ctx.density_of(psi, occ)
    assert np.abs(got - rho).max() < 2e-6 * rho.max()


# every radix of the axis transforms in every step, odd and even lengths, lines that do not fill a
# block, and a grid with a length that has no such form (250: the plane and line-block kernels)
@pytest.mark.parametrize("grid", [(5, 9, 10), (27, 15, 16), (75, 81, 6), (96, 100, 8), (108, 10, 128), (135, 9, 144),
                                  (10, 162, 9), (9, 10, 200), (64, 72, 45), (10, 250, 9)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_grid_transform_lengths(sgo, grid, precision):
    """Both signs against NumPy: 1e-12 of the largest value (float-float keeps 44 bits, 6e-14, through
    fewer than 16 sums a value)."""
    st = dataclasses.replace(workloads.tiny(nat=1, ecut=0.6, kT=0.0, nbands=2), fft=grid)
    ctx = sgo.Context(st, precision=precision, extra_bands=0)
    rng = np.random.default_rng(6)
    x = rng.normal(size=grid) + 1j * rng.normal(size=grid)
    for sign in (-1, 1):
        ref = np.fft.fftn(x) if sign < 0 else np.fft.ifftn(x) * x.size
        assert np.abs(ctx.grid_fft(x, sign) - ref).max() < 1e-12 * np.abs(ref).max()


# members per launch on either side of the eigensolve's cluster rule (8, 4 and 1 CTAs per problem)
@pytest.mark.parametrize("members", [9, 10, 20])
@pytest.mark.parametrize("precision,bands", [("fp64", 9), ("fp64", 40), ("mixed", 130)])
def test_subspace_eigensolve_per_launch(sgo, members, precision, bands):
    """The CTAs of a problem share its work without changing a sum: a member's F and spectrum after a
    few iterations are bitwise those of a batch of two."""
    st = _with_bands(workloads.tiny(nat=2, ecut=9.0, kT=0.01), bands)

    def run(n):
        ctxs = [sgo.Context(st, precision=precision, max_scf=4, autotune=0, sub_batches=1) for _ in range(n)]
        F = sgo.Batch(ctxs).energy_forces()[0]
        return F[0], ctxs[0].eigen()[0]

    two, many = run(2), run(members)
    assert two[0] == many[0]
    assert np.array_equal(two[1], many[1])


# ring lengths of the mixing (a 2 x 2 system, a ring that wraps, the longest), a grid of less than one
# chunk of the reductions and one of several
@pytest.mark.parametrize("hist", [1, 2, 5, 8])
@pytest.mark.parametrize("grid", [(9, 10, 9), (18, 20, 20)])
def test_mixing_history(sgo, hist, grid):
    """The converged F does not depend on the ring's length: second order in the density error of
    1e-7 per electron, so below 1e-9."""
    st = dataclasses.replace(workloads.tiny(nat=2, ecut=1.2, kT=0.01), fft=grid)
    F = [sgo.Context(st, precision="fp64", pulay_hist=h, max_scf=200, scf_tol_rho=1e-7, scf_tol_e=1e-9).energy_forces()[0]
         for h in (hist, 4)]
    assert abs(F[0] - F[1]) < 1e-9


# bands that one lane holds and several, levels far apart and close together against kT
@pytest.mark.parametrize("nbands", [5, 33, 70])
@pytest.mark.parametrize("kT", [1e-4, 0.02, 0.5])
def test_occupations(sgo, nbands, kT):
    """Sum f = N_el (1e-13 N_el is the iteration's rule) and one mu for every partly filled band: from
    f = 2 / (1 + exp(u)), u = ln(2 / f - 1) is known to 2e-16 / (f (2 - f)), 1e-9 kT where f (2 - f) > 1e-6."""
    st = _with_bands(workloads.tiny(nat=2, ecut=6.0, kT=kT), nbands)
    ctx = sgo.Context(st, precision="fp64", max_scf=3, extra_bands=0)
    ctx.energy_forces(check=False)
    eps, occ = ctx.eigen()
    assert abs(occ.sum() - 8.0) < 1e-11
    part = occ * (2.0 - occ) > 1e-6
    mu = (eps - kT * np.log(2.0 / occ.clip(1e-300) - 1.0))[part] if part.any() else np.zeros(1)
    assert np.ptp(mu) < 1e-9 * max(1.0, kT) + 1e-12


def test_autotuner_of_few_tiles(sgo):
    """Two small members have less than a CTA per SM for any number of tiles per rotation CTA: the
    candidates are one launch, and the tuned batch keeps the default on every creation."""
    st = workloads.tiny(nat=2, ecut=6.0)
    for _ in range(8):
        b = sgo.Batch([sgo.Context(st, precision="mixed") for _ in range(2)])
        assert b.tuning()["nn_tc_tiles_per_cta"] == 4
