"""The cooperative kernels' bounded waits running out.

A testing aid (trevr2_debug_set, DEBUG_BARRIER_POLLS) lets a grid barrier poll
once, so that its blocks give up waiting for one another: the kernel returns,
the call reports ETIMEOUT, and nothing the kernel left unfinished is used by
a later call, whose results are those of an undisturbed one, bit for bit."""

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

ETIMEOUT = -4


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
def _aid_off(t2):
    yield
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 0)


def _tree(t2, case):
    return t2.build(case["pos"], case["mass"], case["kappa"], case["lum"], case["h"],
                    case["box_lo"], case["box_size"], case["bucket"])


def _batch(t2, trees, rows):
    return t2.Batch(trees, np.array([0, rows], np.int64), np.array([0], np.int32), nside=2,
                    theta=0.75)


def test_aid_range(t2):
    for v in (-1, (1 << 24) + 1):
        with pytest.raises(t2.TrevrError, match="EINVAL"):
            t2.debug_set(t2.DEBUG_BARRIER_POLLS, v)


@pytest.mark.parametrize("how", ["J", "backward", "prepare", "alpha_table", "batch"])
def test_unfinished_tables_are_not_kept(t2, how):
    case = workloads.random_case(6000, 60, nb=2, seed=401, clumped=True)
    act = case["active"][:900]
    other = _tree(t2, case)
    ref = other.J(act, 2, 0.75)
    ref_alpha = other.alpha_table(2)
    other.free()
    tree = _tree(t2, case)
    held = t2.debug_pool_used()
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 1)
    with pytest.raises(t2.TrevrError, match="absorption tables") as e:
        if how == "J":
            tree.J(act, 2, 0.75)
        elif how == "backward":
            tree.J_backward(act, np.ones((len(act), 2), np.float32), 2, 0.75)
        elif how == "prepare":
            tree.prepare(2)
            tree.status()
        elif how == "alpha_table":
            tree.alpha_table(2)
        else:
            _batch(t2, [tree], len(act))
    assert e.value.code == ETIMEOUT
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 0)
    if how in ("prepare", "alpha_table", "batch"):
        assert t2.debug_pool_used() == held  # J also keeps its walk buffers
    tree.status()  # reported once
    assert torch.equal(tree.J(act, 2, 0.75), ref)
    assert torch.equal(tree.alpha_table(2), ref_alpha)
    plan = _batch(t2, [tree], len(act))
    assert torch.equal(plan.run(torch.as_tensor(act, device="cuda")), ref)
    plan.status()
    plan.free()
    # a table found good before stays when a later one gives up
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 1)
    with pytest.raises(t2.TrevrError, match="absorption tables"):
        tree.J(act, 4, 0.5)
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 0)
    launches = t2.kernel_launches()
    assert torch.equal(tree.J(act, 2, 0.75), ref)
    assert t2.kernel_launches() - launches <= 2  # the walk, its receivers' order
    tree.free()


@pytest.mark.parametrize("flags", ["0", "BUCKET", "backward"])
def test_receiver_order(t2, flags):
    case = workloads.random_case(6000, 60, nb=2, seed=402)
    act = np.random.default_rng(1).integers(0, 6000, size=60_000)
    tree = _tree(t2, case)
    g = np.ones((len(act), 2), np.float32)

    def call():
        if flags == "backward":
            return tree.J_backward(act, g, 2, 0.75)[0]
        return tree.J(act, 2, 0.75, flags=t2.BUCKET if flags == "BUCKET" else 0)

    ref = call()
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 1)
    with pytest.raises(t2.TrevrError, match="receivers' sort") as e:
        call()
    assert e.value.code == ETIMEOUT
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 0)
    if flags == "backward":  # summed with FP32 atomics in any order
        torch.testing.assert_close(call(), ref, rtol=1e-4, atol=1e-6 * float(ref.abs().max()))
    else:
        assert torch.equal(call(), ref)
    tree.free()


@pytest.mark.parametrize("flags", ["0", "BUCKET"])
def test_batch_rows(t2, flags):
    """A batch whose rows were not sorted walks nothing (a tree's range could
    hold another, larger tree's elements): NaN rows and ETIMEOUT."""
    cases = [workloads.random_case(400, 30, nb=2, seed=404),
             workloads.random_case(9000, 60, nb=2, seed=403, clumped=True)]
    trees = [_tree(t2, c) for c in cases]
    rng = np.random.default_rng(2)
    active = torch.as_tensor(np.concatenate([rng.integers(0, 400, size=30_000),
                                             rng.integers(0, 9000, size=50_001)]), device="cuda")
    plan = t2.Batch(trees, np.array([0, 30_000, 80_001], np.int64), np.array([0, 1], np.int32),
                    nside=2, theta=0.75, flags=t2.BUCKET if flags == "BUCKET" else 0)
    ref = plan.run(active)
    plan.status()
    assert bool(torch.isfinite(ref).all())
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 1)
    J = plan.run(active)
    with pytest.raises(t2.TrevrError, match="receivers' sort") as e:
        plan.status()
    assert e.value.code == ETIMEOUT and bool(torch.isnan(J).all())
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 0)
    assert torch.equal(plan.run(active), ref)
    plan.status()
    plan.free()
    for tr in trees:
        tr.free()


# sizes: one block's sort and the cooperative one
@pytest.mark.parametrize("n", [6000, 30_000])
def test_build(t2, n):
    case = workloads.random_case(n, 60, nb=2, seed=405, clumped=True)
    base = t2.debug_pool_used()
    ref = _tree(t2, case)
    perm, B = ref.export("perm"), ref.export("B")
    ref.free()
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 1)
    with pytest.raises(t2.TrevrError, match="gave up waiting") as e:
        _tree(t2, case)
    assert e.value.code == ETIMEOUT and t2.debug_pool_used() == base
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 0)
    tree = _tree(t2, case)
    assert torch.equal(tree.export("perm"), perm) and torch.equal(tree.export("B"), B)
    tree.free()


def test_refusal_costs_no_build(t2):
    """A set outside its cube is refused in about the time of its check and
    sort: its positions are all clamped to one corner, and building that tree
    took one thread 1M additions (634 ms; now 0.45 ms)."""
    n = 1_000_000
    x = torch.rand((n, 3), dtype=torch.float64, device="cuda") + 5.0
    one = torch.ones(n, dtype=torch.float32, device="cuda")
    cols = torch.ones((n, 1), dtype=torch.float32, device="cuda")
    t2.build(x, one, cols, cols, one, box_lo=(5.0, 5.0, 5.0), box_size=1.0).free()
    torch.cuda.synchronize()
    e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    e0.record()
    with pytest.raises(t2.TrevrError, match="outside the given root cube"):
        t2.build(x, one, cols, cols, one, box_lo=(0.0, 0.0, 0.0), box_size=1.0)
    e1.record()
    torch.cuda.synchronize()
    assert e0.elapsed_time(e1) < 100.0


def test_waits_hold_beside_other_work(t2):
    """Cooperative launches beside a walk that fills the GPU, from several threads
    and streams, and in a captured call: none of them waits for blocks that are
    not resident (2^20 polls are a fraction of a second)."""
    import threading
    big = workloads.random_case(30_000, 3000, nb=2, seed=406, clumped=True)
    small = workloads.random_case(20_000, 300, nb=2, seed=407, clumped=True)
    f = [torch.as_tensor(small[k], device="cuda").to(d) for k, d in
         (("pos", torch.float64), ("mass", torch.float32), ("kappa", torch.float32),
          ("lum", torch.float32), ("h", torch.float32))]
    rows = torch.as_tensor(np.random.default_rng(5).integers(0, 20_000, size=30_000), device="cuda")
    walked = _tree(t2, big)
    every = torch.arange(30_000, device="cuda")
    walked.J(every, 8, 0.3)
    ref = t2.build(*f, small["box_lo"], small["box_size"], small["bucket"]).J(rows, 2, 0.75)
    t2.debug_set(t2.DEBUG_BARRIER_POLLS, 1 << 20)
    torch.cuda.synchronize()
    errors = []

    def steps():
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(4):
                    tree = t2.build(*f, small["box_lo"], small["box_size"], small["bucket"], stream=stream)
                    J = tree.J(rows, 2, 0.75, stream=stream)
                    assert torch.equal(J, ref)
                    tree.free()
        except Exception as e:
            errors.append(e)

    long = torch.cuda.Stream()
    for _ in range(4):
        walked.J(every, 8, 0.3, flags=t2.ASYNC, stream=long)
    threads = [threading.Thread(target=steps) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    walked.status()
    tree = t2.build(*f, small["box_lo"], small["box_size"], small["bucket"])
    out = torch.empty_like(ref)
    tree.J(rows, 2, 0.75, out=out)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        tree.J(rows, 2, 0.75, flags=t2.ASYNC, out=out)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    tree.status()
    assert torch.equal(out, ref)
    tree.free()
    walked.free()
