"""The FP64 products in residues (csrc/rns.cu) at the sizes where their tiling
can go wrong, against dense inverses: fronts around the 64-wide panels, the
128-row tiles, the 256-wide blocks and the 480-deep accumulator chunks, rows of
very different scale, non-finite input, and a memory budget that leaves no room
for their scratch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import nao_synth as ns  # noqa: E402
import paper_1405_0194_gb300 as px  # noqa: E402
from oracle import dense  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1405_0194_gb300 import build
    build.build()


def _full(n, seed):
    """A dense symmetric pair on the full pattern (one front of n columns), S diagonally dominant."""
    rng = np.random.default_rng(seed)
    H = rng.standard_normal((n, n)) / np.sqrt(n)
    S = 0.1 * rng.standard_normal((n, n)) / n
    H, S = H + H.T, S + S.T
    S[np.arange(n), np.arange(n)] = 1.0 + np.abs(S).sum(axis=0)
    colptr = np.arange(0, n * n + 1, n, dtype=np.int64)
    rowind = np.tile(np.arange(n, dtype=np.int32), n)
    return colptr, rowind, H, S


def _selinv(n, colptr, rowind, h, s, z, **opts):
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=2, **opts))
    try:
        return px.pexsi_selinv(plan, h, s, z)
    finally:
        px.pexsi_plan_destroy(plan)


# The error of an unpivoted block factorisation at |Im z| = 0.05 with entries of order one: about
# n eps |G|^2 (|G| <= 1 / Im z / lambda_min(S) = 20) < 1e-10, relative to the largest entry.
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 127, 129, 192, 255, 256, 257, 320, 385, 511, 513, 768, 1000])
def test_one_front(n):
    colptr, rowind, H, S = _full(n, n)
    z = 0.1 + 0.05j
    got = _selinv(n, colptr, rowind, H.T.ravel(), S.T.ravel(), z).reshape(n, n).T
    ref = np.linalg.inv(H - z * S)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()


# several atoms of many orbitals in a row: fronts with rows below them, ragged in every size
@pytest.mark.parametrize("norb,atoms", [(37, 9), (70, 9), (131, 7), (150, 6)])
def test_fronts_with_update_sets(norb, atoms):
    s = ns.make_chain(natoms=atoms, seed=norb, norb=norb)
    z = 0.2 + 0.05j
    ref = dense.selected_inverse(s.n, s.colptr, s.rowind, s.H, s.S, z)
    got = _selinv(s.n, s.colptr, s.rowind, s.H, s.S, z, leaf_cols=2 * norb, amalgamate=0)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("n", [64, 65, 200, 257, 600])
def test_inertia_of_one_front(n):
    colptr, rowind, H, S = _full(n, 3 * n)
    shifts = np.array([-0.7, -0.05, 0.3, 1.1])
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=2))
    got = px.pexsi_inertia(plan, H.T.ravel(), S.T.ravel(), shifts)
    px.pexsi_plan_destroy(plan)
    ref = dense.inertia_counts(n, colptr, rowind, H.T.ravel(), S.T.ravel(), shifts)
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("power", [300, -300, 90])
def test_scaled_rows(power):
    """Powers of two: a uniform factor, or one per row and column (D A D), only move exponents in FP64; the
    residue scaling follows the rows, and the inverse has to as well."""
    n = 300
    colptr, rowind, H, S = _full(n, 7)
    z = 0.1 + 0.05j
    ref = np.linalg.inv(H - z * S)
    d = np.full(n, 2.0 ** (power / 2)) if power != 90 else 2.0 ** np.random.default_rng(1).integers(-45, 46, n)
    A = d[:, None] * d[None, :]
    got = _selinv(n, colptr, rowind, (H * A).T.ravel(), (S * A).T.ravel(), z).reshape(n, n).T * A
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()


def test_non_finite_input_is_reported():
    n = 300
    colptr, rowind, H, S = _full(n, 9)
    H[5, 5] = np.nan
    with pytest.raises(px.PexsiError) as e:
        _selinv(n, colptr, rowind, H.T.ravel(), S.T.ravel(), 0.1 + 0.05j)
    assert e.value.code == -5


def test_budget_without_room_for_the_scratch():
    """The smallest budget that a plan accepts leaves no residue scratch; the DFMA kernels then give the same
    inverse to rounding."""
    n = 400
    colptr, rowind, H, S = _full(n, 11)
    z = 0.1 + 0.05j
    h, s = H.T.ravel(), S.T.ravel()
    lo, hi = 1 << 16, 1 << 30
    while hi - lo > 1 << 16:
        mid = (lo + hi) // 2
        try:
            small = _selinv(n, colptr, rowind, h, s, z, hbm_budget=mid)
            hi = mid
        except px.PexsiError as e:
            assert e.code == -3
            lo = mid
    big = _selinv(n, colptr, rowind, h, s, z)
    small = _selinv(n, colptr, rowind, h, s, z, hbm_budget=hi)
    ref = np.linalg.inv(H - z * S).T.ravel()
    assert np.abs(small - ref).max() <= 1e-10 * np.abs(ref).max()
    assert np.abs(big - ref).max() <= 1e-10 * np.abs(ref).max()
    assert not np.array_equal(big, small)  # two different kernels ran


@pytest.mark.parametrize("n", [5, 31, 48, 64])
def test_both_block_inverses_give_the_same_bits(n):
    """Launches of up to 99 block inverses run one on a cluster of CTAs, larger ones one per CTA, with the same
    operations on every entry: a system gives the same bits alone and among 110 others."""
    pats = [_full(n, 100 + k) for k in range(110)]
    host = [px.pexsi_setup(n, p[0], p[1], opts=px.pexsi_opts_default(device=-1)) for p in pats]
    group = px.pexsi_group_create(host, px.pexsi_opts_default(max_batch=1))
    H = [p[2].T.ravel().copy() for p in pats]
    S = [p[3].T.ravel().copy() for p in pats]
    k = len(pats)
    dm, edm, fdm, _ = px.pexsi_group_dm(group, H, S, [0.1] * k, [50.0] * k, 2, [4.0] * k)
    px.pexsi_group_destroy(group)
    plan = px.pexsi_setup(n, pats[0][0], pats[0][1], opts=px.pexsi_opts_default(max_batch=1))
    for q in (0, 57, 109):
        a, b, c, _ = px.pexsi_dm(plan, H[q], S[q], 0.1, 50.0, 2, 4.0)
        assert np.array_equal(a, dm[q]) and np.array_equal(b, edm[q]) and np.array_equal(c, fdm[q])
    px.pexsi_plan_destroy(plan)
    for p in host:
        px.pexsi_plan_destroy(p)


@pytest.mark.parametrize("n", [1, 64, 65, 129, 256, 257, 321, 520])
def test_one_hermitian_front(n):
    """LDU fronts: rows and columns of every product are different operands."""
    colptr, rowind, H, S = _full(n, 5 * n)
    rng = np.random.default_rng(n)
    A, B = rng.standard_normal((n, n)) / np.sqrt(n), 0.05 * rng.standard_normal((n, n)) / n
    H, S = H + 1j * (A - A.T), S + 1j * (B - B.T)
    z = 0.1 + 0.05j
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=2))
    got = px.pexsi_selinv_hermitian(plan, H.T.ravel(), S.T.ravel(), z).reshape(n, n).T
    shifts = np.array([-0.4, 0.2, 0.9])
    counts = px.pexsi_inertia_hermitian(plan, H.T.ravel(), S.T.ravel(), shifts)
    px.pexsi_plan_destroy(plan)
    ref = np.linalg.inv(H - z * S)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()
    ev = np.linalg.eigvalsh(np.linalg.solve(np.linalg.cholesky(S), np.linalg.solve(np.linalg.cholesky(S), H).conj().T))
    assert np.array_equal(counts, [(ev < x).sum() for x in shifts])


# Blocks of 256 columns go into the rest of a front in groups of up to 4: fronts of one block to more than a
# group, whole and ragged, alone and with rows below them, in each kind of factorisation. Bounds as above.
@pytest.mark.parametrize("n", [514, 1024, 1025, 1100, 1281])
def test_grouped_updates_of_one_front(n):
    colptr, rowind, H, S = _full(n, n + 1)
    h, s, z = H.T.ravel(), S.T.ravel(), 0.1 + 0.05j
    got = _selinv(n, colptr, rowind, h, s, z).reshape(n, n).T
    ref = np.linalg.inv(H - z * S)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()
    shifts = np.array([-0.7, 0.3])
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=2))
    counts = px.pexsi_inertia(plan, h, s, shifts)
    A = np.random.default_rng(n).standard_normal((n, n)) / np.sqrt(n)
    Hc = H + 1j * (A - A.T)
    herm = px.pexsi_selinv_hermitian(plan, Hc.T.ravel(), S.T.ravel().astype(complex), z).reshape(n, n).T
    px.pexsi_plan_destroy(plan)
    assert np.array_equal(counts, dense.inertia_counts(n, colptr, rowind, h, s, shifts))
    ref = np.linalg.inv(Hc - z * S)
    assert np.abs(herm - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("norb,leaf", [(290, 600), (270, 1100), (128, 512)])
def test_grouped_updates_with_rows_below(norb, leaf):
    s = ns.make_chain(natoms=6, seed=norb, norb=norb)
    z = 0.2 + 0.05j
    ref = dense.selected_inverse(s.n, s.colptr, s.rowind, s.H, s.S, z)
    got = _selinv(s.n, s.colptr, s.rowind, s.H, s.S, z, leaf_cols=leaf, amalgamate=0)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()


def test_grouped_updates_in_little_scratch():
    """From the least memory that a plan accepts upwards: without the residue scratch, with the least of it, in
    smaller groups and in whole ones, all give the same inverse to rounding."""
    n = 1100
    colptr, rowind, H, S = _full(n, 13)
    h, s, z = H.T.ravel(), S.T.ravel(), 0.1 + 0.05j
    ref = np.linalg.inv(H - z * S).T.ravel()
    budget, seen = 40 << 20, []
    while budget < 1 << 30:
        try:
            got = _selinv(n, colptr, rowind, h, s, z, hbm_budget=int(budget))
            assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()
            if not any(np.array_equal(got, x) for x in seen):
                seen.append(got)
        except px.PexsiError as e:
            assert e.code == -3 and not seen
        budget *= 1.12
    assert len(seen) >= 3
