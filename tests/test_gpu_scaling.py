"""The power-of-two scaling of the FP64 path's matrices (launch_rns_scales): it
may not show in what a call reports or refuses, and it has to find the rows'
sizes wherever they come from."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1405_0194_gb300 as px  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1405_0194_gb300 import build
    build.build()


def _pattern(n):
    return np.arange(0, n * n + 1, n, dtype=np.int64), np.tile(np.arange(n, dtype=np.int32), n)


def _ratio(h, s, mu, beta, table, dE):
    """Smallest |pivot| over the largest entry of the diagonal matrices H - z S of a pole table, |.| = |Re| + |Im|."""
    z = px.pexsi_pole_table(beta, dE, table, mu)["z"]
    a = h[None, :] - z[:, None] * s[None, :]
    a = np.abs(a.real) + np.abs(a.imag)
    return (a.min(axis=1) / a.max(axis=1)).min()


# Pivots of a diagonal matrix are its entries, to the rounding of a multiply-add and of the ratio.
@pytest.mark.parametrize("n", [1, 7, 40, 64])
@pytest.mark.parametrize("blocks", [1, 2])
def test_pivot_ratio_is_the_callers(n, blocks):
    """One block of n columns, inverted on a cluster, or two of them at 64 poles at once (one CTA per inverse)."""
    rng = np.random.default_rng(n)
    d = 2.0 ** -rng.integers(0, 31, n)
    h, s = d * rng.uniform(0.5, 1.5, n), d * rng.uniform(0.8, 1.2, n)
    colptr = np.arange(0, blocks * n * n + 1, n, dtype=np.int64)
    rowind = np.concatenate([np.tile(np.arange(n, dtype=np.int32) + q * n, n) for q in range(blocks)])
    H, S = np.tile(np.diag(h).ravel(), blocks), np.tile(np.diag(s).ravel(), blocks)
    poles = 2 if blocks == 1 else 64
    want = _ratio(h, s, 0.1, 50.0, poles, 4.0)
    plan = px.pexsi_setup(blocks * n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=poles))
    got = px.pexsi_dm(plan, H, S, 0.1, 50.0, poles, 4.0)[3]["min_pivot_ratio"]
    herm = px.pexsi_dm_hermitian(plan, H.astype(complex), S.astype(complex), 0.1, 50.0, poles, 4.0)[3]["min_pivot_ratio"]
    px.pexsi_plan_destroy(plan)
    assert np.allclose([got, herm], want, rtol=1e-13, atol=0)


@pytest.mark.parametrize("others,refused", [(1e-3, False), (1.0, True)])
def test_what_is_refused(others, refused):
    """A level 2^-46 from the shift: a pivot ratio of 1e-11 beside orbitals of 1e-3, of 1e-14 (below the limit of 1e-13)
    beside orbitals of order one. A graded pencil is not refused."""
    n = 60
    colptr, rowind = _pattern(n)
    h, s = np.full(n, 2.0 * others), np.full(n, others)
    h[17], s[17] = 1.0, 1.0
    shift = 1.0 - 2.0 ** -46
    d = 2.0 ** -np.random.default_rng(4).integers(0, 31, n)
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=1))
    try:
        for call, dt in ((px.pexsi_inertia, float), (px.pexsi_inertia_hermitian, complex)):
            H, S = np.diag(h).ravel().astype(dt), np.diag(s).ravel().astype(dt)
            if refused:
                with pytest.raises(px.PexsiError) as e:
                    call(plan, H, S, [shift])
                assert e.value.code == px.capi.PEXSI_ERR_BREAKDOWN
            else:
                assert call(plan, H, S, [shift]).tolist() == [0]
            assert call(plan, np.diag(d * d).ravel().astype(dt), np.diag(d * d).ravel().astype(dt), [0.5]).tolist() == [0]
    finally:
        px.pexsi_plan_destroy(plan)
