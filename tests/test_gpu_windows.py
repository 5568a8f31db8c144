"""Walks whose lists do not hold a receiver's cut at once.

Testing aids (trevr2_debug_set) lower the number of absorbing cells a walk
lists at once and of crossings a warp of a block lists, so that small fields
take the paths of large ones: several windows of cells (with and without
several passes of sources), a full list of crossings, a full stack.

Bars: rows of the per-receiver walks are the undisturbed ones bit for bit (a
source's sums run crossing by crossing however the cells fall into windows);
per-bucket rows and gradients as against the oracle everywhere else (J 1e-4
median, 1e-3 max; the gradients' own bar)."""

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

EINTERNAL = -6


@pytest.fixture(scope="module")
def t2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_15235_gb300 import build_lib
    build_lib.build()
    import paper_2310_15235_gb300 as mod
    mod.load_library()
    return mod


@pytest.fixture(autouse=True)
def _aids_off(t2):
    yield
    for aid in (t2.DEBUG_SOURCE_STACK, t2.DEBUG_CELL_CAP, t2.DEBUG_TEAM_HITS):
        t2.debug_set(aid, 0)


def _tree(t2, case):
    return t2.build(case["pos"], case["mass"], case["kappa"], case["lum"], case["h"],
                    case["box_lo"], case["box_size"], case["bucket"])


def _assert_J(J, ref):
    r = np.abs(J - ref) / np.maximum(np.abs(ref), 1e-300)
    r[(J == 0) & (ref == 0)] = 0.0
    assert np.all(np.isfinite(J)) and np.median(r) <= 1e-4 and r.max() <= 1e-3, (np.median(r), r.max())


def test_aids_reject_bad_settings(t2):
    for what, v in ((t2.DEBUG_CELL_CAP, 33), (t2.DEBUG_CELL_CAP, -32), (t2.DEBUG_TEAM_HITS, -1)):
        with pytest.raises(t2.TrevrError, match="EINVAL"):
            t2.debug_set(what, v)


# sources: fewer than a pass holds, and (2500 at theta 0.4) more; cap 1952 is
# above any cut here: one window
@pytest.mark.parametrize("cap", [32, 64, 224, 1952])
@pytest.mark.parametrize("nside,theta,n_src,nb", [
    (1, 0.45, 200, 2), (2, 0.5, 60, 1), (4, 0.5, 700, 3), (4, 0.4, 2500, 4)])
def test_windows_of_cells(t2, oracle_mod, nside, theta, n_src, nb, cap):
    case = workloads.random_case(3000, n_src, nb=nb, seed=500 + nside, clumped=True)
    tree = _tree(t2, case)
    act = case["active"]
    sub = act[:: max(1, len(act) // 150)]
    plain = {f: tree.J(act, nside, theta, flags=f) for f in (0, t2.SOFT | t2.THICK)}
    ot = oracle_mod.OracleTree.from_case(case)
    if n_src == 2500:  # more than one pass of 1024 sources for some receivers
        assert ot.J(sub, nside, theta, stats=True)[1][:, 3].max() > 1024
    if cap <= 64:
        assert ot.J(sub, nside, theta, stats=True)[1][:, 1].max() > 2 * cap
    t2.debug_set(t2.DEBUG_CELL_CAP, cap)
    for flags, ref in plain.items():
        assert torch.equal(tree.J(act, nside, theta, flags=flags), ref)        # a warp each
        some = torch.as_tensor(sub, device="cuda")
        assert torch.equal(tree.J(sub, nside, theta, flags=flags), ref[some])  # a block each
    plan = t2.Batch([tree], np.array([0, len(sub)], np.int64), np.array([0], np.int32),
                    nside=nside, theta=theta)
    assert torch.equal(plan.run(some), plain[0][some])
    plan.status()
    plan.free()
    for flags in (t2.BUCKET, t2.BUCKET | t2.PP | t2.CSM | t2.THICK):
        want = ot.J(sub, nside, theta, flags=flags)
        _assert_J(tree.J(sub, nside, theta, flags=flags).cpu().numpy(), want)
        plan = t2.Batch([tree], np.array([0, len(sub)], np.int64), np.array([0], np.int32),
                        nside=nside, theta=theta, flags=flags)
        _assert_J(plan.run(some).cpu().numpy(), want)
        plan.status()
        plan.free()
    tree.free()


@pytest.mark.parametrize("nside,theta,n_src,nb", [(2, 0.45, 100, 3), (4, 0.4, 900, 2), (4, 0.4, 2500, 1)])
def test_gradient_windows_of_cells(t2, oracle_mod, nside, theta, n_src, nb):
    import test_gpu_adjoint as adj  # its bar holds here
    case = workloads.random_case(300 if n_src < 2500 else 800, n_src, nb=nb, seed=510 + n_src,
                                 clumped=True, n_active=24)
    tree = _tree(t2, case)
    act = case["active"]
    rng = np.random.default_rng(4)
    gJ = rng.uniform(0.0, 1.0, size=(len(act), nb)).astype(np.float32)
    flags = t2.SOFT | t2.THICK
    ot = oracle_mod.OracleTree.from_case(case)
    assert ot.J(act, nside, theta, stats=True)[1][:, 1].max() > 32
    t2.debug_set(t2.DEBUG_CELL_CAP, 32)
    gk, gl = tree.J_backward(act, gJ, nside, theta, flags=flags)
    ps = adj._all_params(case, n_kappa=100, n_dark=20)
    ps = [ps[i] for i in rng.choice(len(ps), min(len(ps), 300), replace=False)]
    want = adj._oracle_grad(ot, act, gJ.astype(np.float64), nside, theta, ps, flags)
    adj._check(adj._gather(gk, gl, ps), want, f"nside={nside} sources={n_src}")
    tree.free()


@pytest.mark.parametrize("hits", [1, 40, 300])
def test_full_list_of_crossings(t2, hits):
    case = workloads.random_case(3000, 700, nb=3, seed=520, clumped=True)
    tree = _tree(t2, case)
    act = case["active"][:200]
    ref = tree.J(act, 4, 0.5)
    for cap in (0, 96):
        t2.debug_set(t2.DEBUG_CELL_CAP, cap)
        t2.debug_set(t2.DEBUG_TEAM_HITS, hits)
        assert torch.equal(tree.J(act, 4, 0.5), ref)
        t2.debug_set(t2.DEBUG_TEAM_HITS, 0)
    tree.free()


def test_source_stack_overflow_cell_by_cell(t2):
    """As test_source_stack_overflow_is_reported, where the walk goes cell by
    cell: a block and a warp per receiver, per bucket, a plan, the gradient."""
    case = workloads.random_case(2000, 400, nb=2, seed=304, clumped=True)
    tree = _tree(t2, case)
    act = case["active"]
    ref = tree.J(act, 2, 0.5)
    t2.debug_set(t2.DEBUG_SOURCE_STACK, 4)
    calls = [lambda: tree.J(act[:64], 2, 0.5), lambda: tree.J(act, 2, 0.5),
             lambda: tree.J(act, 2, 0.5, flags=t2.BUCKET),
             lambda: tree.J_backward(act[:64], np.ones((64, 2), np.float32), 2, 0.5)]
    plan = t2.Batch([tree], np.array([0, 64], np.int64), np.array([0], np.int32), nside=2, theta=0.5)
    calls.append(lambda: (plan.run(torch.as_tensor(act[:64], device="cuda")), plan.status()))
    for call in calls:
        with pytest.raises(t2.TrevrError, match="stack overflow") as e:
            call()
        assert e.value.code == EINTERNAL
    plan.free()
    t2.debug_set(t2.DEBUG_SOURCE_STACK, 0)
    tree.status()
    assert torch.equal(tree.J(act, 2, 0.5), ref)
    tree.free()
