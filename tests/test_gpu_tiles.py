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
