"""The edges between the library's paths: where a dispatch rule changes the
kernel (cooperative or one-block sort and topology, cell by cell or beam by
beam, a block or a warp per receiver, sources in one or several windows), the
result has to be the same tree and the same J.

Bars: trees bit-exact against the oracle; J within 1e-4 (median) and 1e-3 (max)
of the oracle, as for every other walk; rows of the same receivers bit-equal
however many are asked for."""

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def t2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_15235_gb300 import build_lib
    build_lib.build()
    import paper_2310_15235_gb300 as mod
    mod.load_library()
    return mod


def _tree(t2, case, **kw):
    box = dict(box_lo=case["box_lo"], box_size=case["box_size"])
    box.update(kw)
    return t2.build(case["pos"], case["mass"], case["kappa"], case["lum"], case["h"],
                    bucket=case["bucket"], **box)


def _assert_J(J, ref):
    r = np.abs(J - ref) / np.maximum(np.abs(ref), 1e-300)
    r[(J == 0) & (ref == 0)] = 0.0
    assert np.all(np.isfinite(J)) and np.median(r) <= 1e-4 and r.max() <= 1e-3, (np.median(r), r.max())


# sizes around the one-block sort (8192), the first level of more than 1024
# nodes, chunks of 2048 keys; bucket 1 outgrows the first node arrays
@pytest.mark.parametrize("n,bucket,clumped", [
    (2, 1, False), (8192, 12, True), (8193, 12, False), (20_481, 1, True), (70_000, 3, True)])
def test_sort_and_topology(t2, oracle_mod, n, bucket, clumped):
    case = workloads.random_case(n - 1, 1, nb=1, seed=n, clumped=clumped, bucket=bucket)
    if clumped:
        case["pos"][: n // 100] = case["pos"][0]  # equal keys keep the caller's order
    tree = _tree(t2, case)
    e = oracle_mod.OracleTree.from_case(case).export()
    np.testing.assert_array_equal(tree.export("perm").cpu().numpy(), e["perm"])
    for f in ("prefix", "depth", "first", "count", "child", "parent"):
        got = tree.export(f).cpu().numpy()
        got = got.view(np.uint64) if f == "prefix" else got
        np.testing.assert_array_equal(got.astype(e[f].dtype), e[f], err_msg=f)
    tree.free()


def test_root_cube(t2):
    """The bounding cube, and an edge whose reciprocal is not exact."""
    case = workloads.random_case(9000, 9, nb=2, seed=5)
    lo = case["pos"].min(0)
    tree = _tree(t2, case, box_lo=None, box_size=0.0)
    assert tree.box_lo == tuple(lo) and tree.box_size == (case["pos"].max(0) - lo).max()
    tree.free()
    cube = _tree(t2, case, box_lo=(-0.1, -0.1, -0.1), box_size=1.3)
    u = np.floor((case["pos"] + 0.1) / 1.3 * 2.0 ** 21).astype(np.uint64)
    keys = np.zeros(len(u), np.uint64)
    for bit in range(21):
        for a in range(3):
            keys |= ((u[:, a] >> np.uint64(bit)) & np.uint64(1)) << np.uint64(3 * bit + 2 - a)
    np.testing.assert_array_equal(cube.export("keys").cpu().numpy().view(np.uint64), np.sort(keys))
    cube.free()


# theta and the number of sources on both sides of the rule, every band count;
# 2500 sources: several windows of sources per walk
@pytest.mark.parametrize("nside,theta,n_src,nb", [
    (1, 0.45, 4, 1), (1, 0.75, 3, 2), (2, 0.45, 16, 3), (2, 0.44, 16, 4), (2, 0.75, 15, 1),
    (4, 0.4, 64, 2), (4, 0.6, 63, 3), (4, 0.6, 64, 4), (4, 0.5, 2500, 3), (8, 0.6, 200, 2)])
def test_cells_and_beams(t2, oracle_mod, nside, theta, n_src, nb):
    case = workloads.random_case(3000, n_src, nb=nb, seed=nside * 100 + n_src, clumped=n_src > 60)
    act = case["active"][:: max(1, len(case["active"]) // 200)]
    tree = _tree(t2, case)
    ot = oracle_mod.OracleTree.from_case(case)
    for flags in (0, t2.BUCKET, t2.BUCKET | t2.PP | t2.CSM):
        if flags & t2.PP and nside > 4:
            continue  # spheres beyond the particles a walk holds
        _assert_J(tree.J(act, nside, theta, flags=flags).cpu().numpy(),
                  ot.J(act, nside, theta, flags=flags))
    tree.free()


@pytest.mark.parametrize("nside,theta,edge", [(2, 0.75, 640), (4, 0.5, 1024)])
def test_rows_do_not_depend_on_how_many_are_asked(t2, nside, theta, edge):
    case = workloads.random_case(9000, 1800, nb=3, seed=nside, clumped=True)
    tree = _tree(t2, case)
    full = tree.J(case["active"], nside, theta)
    rng = np.random.default_rng(1)
    for A in (1, 31, edge, edge + 1, 8192, 8193):
        sub = rng.choice(len(case["active"]), size=A, replace=A > 8192)  # any order, repeats
        J = tree.J(case["active"][sub], nside, theta)
        assert torch.equal(J, full[torch.as_tensor(sub, device=J.device)]), A
    with pytest.raises(t2.TrevrError, match="EINVAL"):
        tree.J(np.array([0, len(case["pos"]), 5]), nside, theta)
    tree.free()


# the gradient on both sides of the same rule; 900 sources: two windows per
# pass, 2500: two passes (1683 sources of a receiver at most)
@pytest.mark.parametrize("nside,theta,n_src,nb", [
    (1, 0.45, 4, 1), (2, 0.45, 16, 3), (2, 0.45, 15, 3), (2, 0.44, 16, 2), (4, 0.4, 64, 4),
    (4, 0.4, 900, 2), (4, 0.4, 2500, 1)])
def test_gradient_cells_and_beams(t2, oracle_mod, nside, theta, n_src, nb):
    import test_gpu_adjoint as adj  # its bar holds here
    case = workloads.random_case(300 if n_src > 64 else 800, n_src, nb=nb,
                                 seed=nside * 100 + n_src, clumped=n_src > 60, n_active=24)
    tree = _tree(t2, case)
    act = case["active"]
    rng = np.random.default_rng(3)
    gJ = rng.uniform(0.0, 1.0, size=(len(act), nb)).astype(np.float32)
    flags = t2.SOFT | t2.THICK
    gk, gl = tree.J_backward(act, gJ, nside, theta, flags=flags)
    ps = adj._all_params(case, n_kappa=100, n_dark=20)
    ps = [ps[i] for i in rng.choice(len(ps), min(len(ps), 300), replace=False)]
    want = adj._oracle_grad(oracle_mod.OracleTree.from_case(case), act, gJ.astype(np.float64),
                            nside, theta, ps, flags)
    adj._check(adj._gather(gk, gl, ps), want, f"nside={nside} sources={n_src}")
    tree.free()


def test_short_rungs_of_many_sources(t2):
    """Receivers with more sources than a pass holds: a block for each gives the
    rows of a warp for each (as a plan walks them), in clearly less time.  When
    such receivers were left to one of the block's warps it took the same time."""
    case = workloads.random_case(100_000, 200_000, nb=2, seed=12, clumped=True)
    tree = _tree(t2, case)
    act = torch.as_tensor(np.random.default_rng(3).choice(100_000, 300, replace=False), device="cuda")
    plan = t2.Batch([tree], np.array([0, 300], np.int64), np.array([0], np.int32), nside=4, theta=0.5)

    def ms(run):
        best = np.inf
        for _ in range(8):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            J = run()
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best, J

    block, J = ms(lambda: tree.J(act, 4, 0.5))
    warp, ref = ms(lambda: plan.run(act))
    plan.status()
    assert torch.equal(J, ref)
    assert block <= 0.75 * warp, (block, warp)
    plan.free()
    tree.free()


@pytest.mark.parametrize("nside,theta", [(1, 0.5), (2, 0.75), (4, 0.5), (4, 0.3), (8, 0.6)])
def test_prepare_leaves_nothing_to_the_first_call(t2, nside, theta):
    """After trevr2_prepare the first J launches what a later one does."""
    case = workloads.random_case(3000, 300, nb=1, seed=13)
    tree = _tree(t2, case)
    tree.prepare(nside)
    launches = [t2.kernel_launches()]
    for _ in range(2):
        tree.J(case["active"], nside, theta)
        launches.append(t2.kernel_launches())
    assert launches[1] - launches[0] == launches[2] - launches[1]
    tree.free()


@pytest.mark.parametrize("n,bucket", [(20_000, 1), (9000, 2), (1500, 1)])
def test_topology_outgrows_its_arrays(t2, oracle_mod, n, bucket):
    """Elements on a line split along one axis of three, so the tree has more nodes
    than the arrays it is first built into (4 n / bucket + 64): built again into
    larger ones, from a level all blocks share (20,000; 9,000) or block 0's."""
    case = workloads.random_case(n - 1, 1, nb=1, seed=n, bucket=bucket)
    case["pos"][:, 1:] = 0.375
    e = oracle_mod.OracleTree.from_case(case).export()
    first = max(1024, 4 * (n // bucket) + 64)
    assert len(e["depth"]) > first
    full = np.searchsorted(np.cumsum(np.bincount(e["depth"])), first, side="right")  # its level
    assert (np.bincount(e["depth"])[full - 1] > 1024) == (n > 1500)
    tree = _tree(t2, case)
    np.testing.assert_array_equal(tree.export("perm").cpu().numpy(), e["perm"])
    for f in ("prefix", "depth", "first", "count", "child", "parent"):
        got = tree.export(f).cpu().numpy()
        got = got.view(np.uint64) if f == "prefix" else got
        np.testing.assert_array_equal(got.astype(e[f].dtype), e[f], err_msg=f)
    tree.free()
