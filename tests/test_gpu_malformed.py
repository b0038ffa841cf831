"""Malformed runs in the allocation-free batch: a function that finds one
operand instead of two is refused wherever it stands, also when a leaf to its
left leaves one value at the end, and the trees beside it are evaluated."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _call(trees, C):
    import torch
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    x, t = synth.cases(11, C)
    k = synth.consts(11)
    off = np.concatenate([[0], np.cumsum([len(s) for s in trees])]).astype(np.int64)
    ops = np.concatenate([np.asarray(s, np.uint8) for s in trees])
    dev = torch.device("cuda", 0)
    d_ops = torch.zeros((len(ops) + 15) // 16 * 16, dtype=torch.uint8, device=dev)
    d_ops[:len(ops)] = torch.from_numpy(ops).to(dev)
    d = [torch.from_numpy(np.ascontiguousarray(v)).to(dev) for v in (off, x, t, np.asarray(k, np.float32))]
    vals = torch.full((len(trees), C), float("nan"), device=dev)
    fit = torch.full((len(trees),), float("nan"), device=dev)
    try:
        flags = gp.gp_eval_small_noalloc(d_ops, *d, vals, fit)
    except gp.GpError as e:
        assert e.code == gp.GP_EINVAL and "0x2" in str(e), e
        flags = 2
    return flags, vals.cpu().numpy(), (x, t, k)


def _right_comb(n):
    return [0, 4] * n + [4]


@pytest.mark.parametrize("C", [7, 48, 300])
def test_a_function_with_one_operand_is_refused(C):
    """[x, +] before a whole tree of n nodes: one value is complete, + takes it and what was there before, x follows.
    The sizes put that function at every byte of a word and on both sides of a chunk's edge."""
    assert _call([[4, 0, 0, 4, 4]], C)[0] == 2
    for shift in range(4):                            # where the tree starts within its word
        for n in list(range(3, 20, 2)) + [121, 123, 125, 127, 129, 251, 253, 255, 257, 1001]:
            bad = [4, 0] + _right_comb(n // 2)
            assert _call([[4]] * shift + [bad], C)[0] == 2, (shift, n)


@pytest.mark.parametrize("bad", [[0], [4, 4], [0, 4], [0, 0, 4], [4, 0, 4], [4, 0, 4, 0, 4, 4], [0, 4, 0, 0, 4, 4],
                                 [4, 0, 0, 0, 4, 4, 4]])
def test_other_malformed_runs(bad):
    assert _call([bad], 48)[0] == 2


def test_trees_beside_a_malformed_one():
    import oracle
    good = [_right_comb(n) for n in (0, 1, 2, 61, 62, 63, 64, 65, 126, 127, 128, 400)]
    flags, vals, (x, t, k) = _call(good, 100)
    assert flags == 0
    flags, mixed, _ = _call(good[:6] + [[4, 0, 0, 4, 4]] + good[6:], 100)
    assert flags == 2
    assert np.array_equal(np.delete(mixed, 6, 0), vals)
    off = np.concatenate([[0], np.cumsum([len(s) for s in good])]).astype(np.uint64)
    ov, _ = oracle.eval_pop_f32(np.concatenate([np.asarray(s, np.uint8) for s in good]), off, k, x, t)
    assert np.array_equal(oracle.canon_nan(vals), oracle.canon_nan(ov))
