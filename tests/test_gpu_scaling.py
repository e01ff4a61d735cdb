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


def _h0(n, seed, pairs=False):
    """Symmetric with eigenvalues of 0.8 to 2.2 in size: +-1.5 on the diagonal (pairs: 1.5 beside a zero diagonal in
    every third pair of columns) and a random part of norm 0.7."""
    rng = np.random.default_rng(seed)
    G = rng.standard_normal((n, n))
    H = 0.25 * (G + G.T) / np.sqrt(n)
    d = np.where(rng.random(n) < 0.5, -1.5, 1.5)
    for k in range(0, n - 1, 6) if pairs else ():
        H[k, k] = H[k + 1, k + 1] = d[k] = d[k + 1] = 0.0
        H[k, k + 1] = H[k + 1, k] = 1.5
    return H + np.diag(d)


def _graded(kind, n):
    """H, S, the shift and the scaling under which H - z S has a condition number below 10."""
    rng = np.random.default_rng(5)
    c = np.arange(n)
    if kind == "overlap":  # a large shift and an uneven overlap
        e = 2.0 ** -rng.integers(0, 18, n)
        return _h0(n, 1), np.diag(e * e), 2.0 ** 40 * (1 + 1j), 2.0 ** -20 / e
    if kind == "level":  # a panel of levels at the shift with weak couplings
        d = np.where(c // 64 == 1, 2.0 ** -40, 1.0)
        return d[:, None] * _h0(n, 2) * d + 0.25 * np.eye(n), np.eye(n), 0.25 + 2.0 ** -80 * 1j, 1 / d
    z = 2.0 ** -40 * (1 + 1j)
    if kind == "zeros":
        return _h0(n, 3, pairs=True), np.eye(n), z, np.ones(n)
    d = 2.0 ** -rng.integers(0, 18, n) if kind == "rows" else 2.0 ** (-15.0 * (c // 64 % 4))
    return d[:, None] * _h0(n, 4) * d, np.eye(n), z, 1 / np.maximum(d, 2.0 ** -20)


# Forward error of the scaled matrix in FP64: n eps times the square of its condition number (100), n = 300: 7e-12.
@pytest.mark.parametrize("hermitian", [False, True])
@pytest.mark.parametrize("kind", ["rows", "panels", "overlap", "level", "zeros"])
def test_graded_matrices(kind, hermitian):
    """H of very different rows beside S = I (or S of such rows beside H): the inverse is accurate to the rows' sizes."""
    n = 300
    H, S, z, scale = _graded(kind, n)
    A = scale[:, None] * (H - z * S) * scale
    assert np.linalg.cond(A) < 10
    colptr, rowind = _pattern(n)
    plan = px.pexsi_setup(n, colptr, rowind, perm=np.arange(n, dtype=np.int32), opts=px.pexsi_opts_default(max_batch=2))
    s = None if np.array_equal(S, np.eye(n)) else S.ravel()
    if hermitian:
        s = None if s is None else s.astype(complex)
        got = px.pexsi_selinv_hermitian(plan, H.ravel().astype(complex), s, z)
    else:
        got = px.pexsi_selinv(plan, H.ravel(), s, z)
    if kind in ("rows", "panels", "zeros"):
        counts = (px.pexsi_inertia_hermitian(plan, H.ravel().astype(complex), s, [0.0]) if hermitian
                  else px.pexsi_inertia(plan, H.ravel(), s, [0.0]))
        d = scale if kind != "panels" else 2.0 ** (15.0 * (np.arange(n) // 64 % 4))
        assert counts.tolist() == [int((np.linalg.eigvalsh(d[:, None] * H * d) < 0).sum())]
    px.pexsi_plan_destroy(plan)
    ref = np.linalg.inv(A)
    err = np.abs(got.reshape(n, n) / scale[:, None] / scale - ref).max() / np.abs(ref).max()
    assert err <= 7e-12, err


def test_scaling_follows_each_shift():
    """Shifts of very different size in one batch give the bits that each gives alone, and counts as in 64 bits."""
    n = 200
    colptr, rowind = _pattern(n)
    d = 2.0 ** -np.random.default_rng(8).integers(0, 18, n)
    H = d[:, None] * _h0(n, 9) * d
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=4))
    shifts = [-2.0 ** 30, -4.0, 0.0, 2.0 ** -60, 4.0]
    counts = px.pexsi_inertia(plan, H.ravel(), None, shifts)
    assert counts.tolist() == [0, 0, *[int((np.linalg.eigvalsh(H / d[:, None] / d) < 0).sum())] * 2, n]
    both = px.pexsi_dm(plan, H.ravel(), None, 0.0, 1e6, 4, 4.0)[0]
    one = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=1))
    alone = px.pexsi_dm(one, H.ravel(), None, 0.0, 1e6, 4, 4.0)[0]
    for p in (plan, one):
        px.pexsi_plan_destroy(p)
    assert np.abs(both - alone).max() <= 1e-13 * np.abs(alone).max()  # the same inverses, added up in another order


# Entry by entry: rounding every operation of an elimination without growth leaves |dG| <= n eps |G| |A| |G|; as much again
# for the reference.
@pytest.mark.parametrize("kind", ["chain", "fluid", "sheet"])
@pytest.mark.parametrize("overlap", [True, False])
def test_entries_of_ordinary_systems(kind, overlap):
    """The operands are rounded against their rows' norms; on the patterns of such systems every entry of the inverse is
    still accurate to its own size."""
    import nao_synth as ns
    s = {"chain": ns.make_chain, "fluid": lambda: ns.make_fluid(nmol=24), "sheet": lambda: ns.make_sheet(ncell=6)}[kind]()
    cols = np.repeat(np.arange(s.n), np.diff(s.colptr))
    A, z = np.zeros((s.n, s.n), complex), 0.1 + 0.01j
    A[s.rowind, cols] = s.H - z * (s.S if overlap else (s.rowind == cols))
    plan = px.pexsi_setup(s.n, s.colptr, s.rowind, opts=px.pexsi_opts_default(max_batch=1))
    got = px.pexsi_selinv(plan, s.H, s.S if overlap else None, z)
    px.pexsi_plan_destroy(plan)
    G = np.linalg.inv(A)
    bound = 2 * s.n * np.finfo(float).eps * (np.abs(G) @ np.abs(A) @ np.abs(G))
    assert (np.abs(got - G[s.rowind, cols]) <= bound[s.rowind, cols]).all()
