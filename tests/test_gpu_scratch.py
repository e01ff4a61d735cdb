"""The scratch of the FP64 path's residue products: what is chosen for a plan, and
that results do not follow the batch or the fronts that run beside one."""
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


def _blocks(sizes, seed):
    """Independent dense symmetric pairs side by side (a front each), S diagonally dominant."""
    colptr, rowind, H, S, at = [np.zeros(1, np.int64)], [], [], [], 0
    for n in sizes:
        rng = np.random.default_rng(seed + n)
        h = rng.standard_normal((n, n)) / np.sqrt(n)
        s = 0.1 * rng.standard_normal((n, n)) / n
        h, s = h + h.T, s + s.T
        s[np.arange(n), np.arange(n)] = 1.0 + np.abs(s).sum(axis=0)
        colptr.append(colptr[-1][-1] + n * np.arange(1, n + 1, dtype=np.int64))
        rowind.append(np.tile(np.arange(at, at + n, dtype=np.int32), n))
        H.append(h.ravel())
        S.append(s.ravel())
        at += n
    return at, np.concatenate(colptr), np.concatenate(rowind), np.concatenate(H), np.concatenate(S)


def _inverses(system, max_batch):
    n, colptr, rowind, H, S = system
    plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(max_batch=max_batch))
    got = px.pexsi_selinv(plan, H, S, 0.1 + 0.05j)
    herm = px.pexsi_selinv_hermitian(plan, H.astype(complex), S.astype(complex), 0.1 + 0.05j)
    px.pexsi_plan_destroy(plan)
    return got, herm


# 600 to 2200: fronts of more than a block of 256 columns, up to more than two groups of four
@pytest.mark.parametrize("n", [600, 1100, 2200])
def test_bits_do_not_follow_the_batch(n):
    system = _blocks([n], 1)
    ref = _inverses(system, 1)
    for batch in (2, 4, 8):
        for a, b in zip(ref, _inverses(system, batch)):
            assert np.array_equal(a, b)


def test_bits_do_not_follow_the_neighbours():
    alone = _inverses(_blocks([700], 1), 1)
    beside = _inverses(_blocks([1100, 700, 300], 1), 2)
    for a, b in zip(alone, beside):
        assert np.array_equal(a, b[1100 * 1100:1100 * 1100 + 700 * 700])


@pytest.mark.parametrize("kind", ["chain", "sheet", "blocks"])
def test_batch_under_a_budget(kind):
    """A fifth more than the workspace that eight poles take with all the scratch they want (the budget also counts what
    other calls allocate later) holds at least eight of an automatic batch, half of it at least three, and nothing exceeds
    a budget."""
    import nao_synth as ns
    if kind == "blocks":
        n, colptr, rowind, H, S = _blocks([300, 300, 200], 2)
    else:
        s = ns.make_chain(natoms=300) if kind == "chain" else ns.make_sheet(ncell=8)
        n, colptr, rowind, H, S = s.n, s.colptr, s.rowind, s.H, s.S

    def chosen(**opts):
        plan = px.pexsi_setup(n, colptr, rowind, opts=px.pexsi_opts_default(**opts))
        try:
            px.pexsi_selinv(plan, H, S, 0.1 + 0.05j)
            st = px.pexsi_plan_get_stats(plan)
            return st["batch"], st["workspace_bytes"]
        except px.PexsiError as e:
            assert e.code == -3
            return 0, 0
        finally:
            px.pexsi_plan_destroy(plan)

    _, eight = chosen(max_batch=8)
    for x in (0.02, 0.1, 0.2, 0.35, 0.6, 0.8, 1.2, 2.0, 4.0):
        batch, used = chosen(hbm_budget=int(x * eight))
        assert used <= int(x * eight)
        assert batch >= (8 if x >= 1.2 else 3 if x >= 0.6 else 0)
