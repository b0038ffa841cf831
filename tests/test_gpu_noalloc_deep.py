"""Trees deeper than a warp's stack window in the allocation-free batch: fewer
and more of them than overflow stacks, alone and among shallow ones, over one
and many case blocks, against the CPU oracle bit for bit (the same operations
on the same operands)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _comb(n, rng):
    """n functions, then n + 1 leaves: n + 1 values wait at once."""
    return np.concatenate([rng.integers(0, 4, n), rng.integers(4, 256, n + 1)]).astype(np.uint8)


def _run(trees, C):
    import torch
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    x, t = synth.cases(8, C)
    k = synth.consts(8)
    off = np.concatenate([[0], np.cumsum([len(s) for s in trees])]).astype(np.int64)
    ops = np.concatenate(trees)
    dev = torch.device("cuda", 0)
    d_ops = torch.zeros((len(ops) + 15) // 16 * 16, dtype=torch.uint8, device=dev)
    d_ops[:len(ops)] = torch.from_numpy(ops).to(dev)
    d = [torch.from_numpy(np.ascontiguousarray(v)).to(dev) for v in (off, x, t, np.asarray(k, np.float32))]
    vals = torch.full((len(trees), C), float("nan"), device=dev)
    fit = torch.full((len(trees),), float("nan"), device=dev)
    flags = 0
    try:
        flags = gp.gp_eval_small_noalloc(d_ops, *d, vals, fit)
    except gp.GpError as e:
        assert e.code == gp.GP_EINVAL and "0x2" in str(e), e
        flags = 2
    return flags, vals.cpu().numpy(), fit.cpu().numpy(), (ops, off.astype(np.uint64), k, x, t)


@pytest.mark.parametrize("C", [1, 32, 33, 100, 4096])
@pytest.mark.parametrize("deep,shallow", [(1, 0), (2, 3), (63, 0), (64, 1), (65, 200), (129, 0), (1000, 1000)])
def test_deep_trees(deep, shallow, C):
    import oracle
    if deep * C > 500_000:
        pytest.skip("the oracle's share of the time")
    rng = np.random.default_rng(deep * 7 + shallow)
    # one entry below, at and above the windows of 48 and 96 entries, and the deepest tree there is
    trees = [_comb((511, 46, 47, 48, 49, 94, 95, 96, 97, 200)[j % 10], rng) for j in range(deep)]
    trees += [_comb(int(rng.integers(0, 20)), rng) for _ in range(shallow)]
    trees = [trees[j] for j in rng.permutation(len(trees))]
    flags, vals, fit, (ops, off, k, x, t) = _run(trees, C)
    assert flags == 0
    ov, of = oracle.eval_pop_f32(ops, off, k, x, t)
    assert np.array_equal(oracle.canon_nan(vals), oracle.canon_nan(ov))
    assert np.array_equal(oracle.canon_nan(fit), oracle.canon_nan(of))


@pytest.mark.parametrize("C", [20, 200])
def test_a_malformed_deep_tree_among_others(C):
    import oracle
    rng = np.random.default_rng(5)
    good = [_comb(int(n), rng) for n in rng.integers(1, 400, 150)]
    bad = np.concatenate([np.array([4, 0], np.uint8), _comb(300, rng)])
    flags, vals, fit, (ops, off, k, x, t) = _run(good[:70] + [bad] + good[70:], C)
    assert flags == 2
    flags, _, _, (ops, off, k, x, t) = _run(good, C)
    assert flags == 0
    ov, of = oracle.eval_pop_f32(ops, off, k, x, t)
    assert np.array_equal(oracle.canon_nan(np.delete(vals, 70, 0)), oracle.canon_nan(ov))
    assert np.array_equal(oracle.canon_nan(np.delete(fit, 70)), oracle.canon_nan(of))
