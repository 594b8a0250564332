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
