"""Waits of the FP64 path that run out, made to happen without faulting the GPU
(pexsi_opts.inject = 1, wait_ns = 2 ms): the launch ends cleanly, the call
returns PEXSI_ERR_TIMEOUT and names the wait, and the context stays usable.

A front of up to 64 columns without rows below it runs the block inverse and no
GEMM, so its timeout is the block inverse's: the first column of the cluster
comes 8 ms late. Where the block inverses run one to a CTA, which does not wait,
the timeout is the residue GEMM's: its CTA 0 copies no operands.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1405_0194_gb300 as px  # noqa: E402

WAIT_NS = 2_000_000


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1405_0194_gb300 import build
    build.build()


def _full(n, seed):
    """A dense symmetric pair on the full pattern (one front of n columns)."""
    rng = np.random.default_rng(seed)
    H = rng.standard_normal((n, n)) / np.sqrt(n)
    H = H + H.T
    S = np.eye(n)
    return np.arange(0, n * n + 1, n, dtype=np.int64), np.tile(np.arange(n, dtype=np.int32), n), H, S


def _times_out(call, what):
    with pytest.raises(px.PexsiError) as e:
        call()
    assert e.value.code == px.capi.PEXSI_ERR_TIMEOUT
    assert what in str(e.value) and "wait ran out" in str(e.value)


def _works(n, colptr, rowind, H, S):
    torch.cuda.synchronize()  # no sticky error: the launches returned normally
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=2, wait_ns=500_000_000))
    got = px.pexsi_selinv(plan, H.ravel(), S.ravel(), 0.1 + 0.05j).reshape(n, n)
    px.pexsi_plan_destroy(plan)
    ref = np.linalg.inv(H - (0.1 + 0.05j) * S)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("n", [1, 13, 48, 64])
def test_block_inverse(n):
    colptr, rowind, H, S = _full(n, n)
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=2, inject=1, wait_ns=WAIT_NS))
    try:
        _times_out(lambda: px.pexsi_selinv(plan, H.ravel(), S.ravel(), 0.1 + 0.05j), "block inverse")
        _times_out(lambda: px.pexsi_dm(plan, H.ravel(), S.ravel(), 0.1, 50.0, 2, 4.0), "block inverse")
        _times_out(lambda: px.pexsi_inertia(plan, H.ravel(), S.ravel(), [0.1, 0.2]), "block inverse")
        Hc = H.ravel().astype(complex)
        _times_out(lambda: px.pexsi_selinv_hermitian(plan, Hc, S.ravel().astype(complex), 0.1 + 0.05j), "block inverse")
        _times_out(lambda: px.pexsi_inertia_hermitian(plan, Hc, S.ravel().astype(complex), [0.1]), "block inverse")
    finally:
        px.pexsi_plan_destroy(plan)
    _works(n, colptr, rowind, H, S)


def test_residue_gemm():
    """Two fronts of 300 columns for 64 poles at once: more than 99 block inverses a launch, which run one to a CTA without
    waits, so that the timeout is the GEMM's."""
    n = 300
    colptr, rowind, H, S = _full(n, n)
    colptr = np.concatenate([colptr, colptr[-1] + colptr[1:]])
    rowind = np.concatenate([rowind, rowind + n])
    h, s = np.tile(H.ravel(), 2), np.tile(S.ravel(), 2)
    plan = px.pexsi_setup(2 * n, colptr, rowind.astype(np.int32),
                          opts=px.pexsi_opts_default(max_batch=64, inject=1, wait_ns=WAIT_NS))
    try:
        _times_out(lambda: px.pexsi_dm(plan, h, s, 0.1, 50.0, 64, 4.0), "tensor-core GEMM")
        _times_out(lambda: px.pexsi_inertia(plan, h, s, np.linspace(0.1, 0.2, 64)), "tensor-core GEMM")
        _times_out(lambda: px.pexsi_dm_hermitian(plan, h.astype(complex), s.astype(complex), 0.1, 50.0, 64, 4.0),
                   "tensor-core GEMM")
    finally:
        px.pexsi_plan_destroy(plan)
    _works(n, *_full(n, n))


@pytest.mark.parametrize("n", [33, 64])
def test_cluster_inverses_repeat_their_bits(n):
    """The staged pivot column is read by every lane of the search warp before the next one replaces it: the inverses of
    many launches, with row interchanges in nearly every step, are the same bits each time."""
    colptr, rowind, H, S = _full(n, 7 * n)
    Hc = (H + 1j * (np.triu(H, 1) - np.tril(H, -1))).T.ravel()
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=2))
    first = px.pexsi_selinv(plan, H.ravel(), S.ravel(), 0.1 + 0.05j)
    herm = px.pexsi_selinv_hermitian(plan, Hc, S.ravel().astype(complex), 0.1 + 0.05j)
    for _ in range(60):
        assert np.array_equal(first, px.pexsi_selinv(plan, H.ravel(), S.ravel(), 0.1 + 0.05j))
        assert np.array_equal(herm, px.pexsi_selinv_hermitian(plan, Hc, S.ravel().astype(complex), 0.1 + 0.05j))
    px.pexsi_plan_destroy(plan)
