"""A batch of deep trees keeps most warps waiting for an overflow stack until
nearly its end.  The wait's bound is against a stack that never comes free, not
against a long batch: with a bound far below the batch's time (a copy of the
source compiled with another constant) every tree is still evaluated."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _library(tmp_path, polls):
    from paper_2205_03251_gb300 import _build
    src = open(os.path.join(_build.CSRC, "noalloc.cu")).read()
    src, n = re.subn(r"NA_SPIN = 1u << \d+", f"NA_SPIN = {polls}u", src)
    assert n == 1
    (tmp_path / "noalloc.cu").write_text(src)
    lib = tmp_path / "libnoalloc.so"
    subprocess.check_call([_build._nvcc(), *_build.NVCC_FLAGS, "-I", _build.INCLUDE, "-I", _build.CSRC, "-o", str(lib),
                           str(tmp_path / "noalloc.cu")])
    return ctypes.CDLL(str(lib))


def test_the_bound_counts_from_the_last_turn(tmp_path):
    """One tree takes a warp about 0.37 ms, 4,096 polls some milliseconds, the batch about 23 ms."""
    import torch
    import oracle
    import synth
    lib = _library(tmp_path, 4096)
    P, C = 4000, 100
    rng = np.random.default_rng(1)
    tree = np.concatenate([rng.integers(0, 4, 511), rng.integers(4, 256, 512)]).astype(np.uint8)
    x, t = synth.cases(8, C)
    k = np.asarray(synth.consts(8), np.float32)
    dev = torch.device("cuda", 0)
    ops = np.zeros((P * 1023 + 15) // 16 * 16, np.uint8)
    ops[:P * 1023] = np.tile(tree, P)
    off = np.arange(P + 1, dtype=np.int64) * 1023
    d = [torch.from_numpy(v).to(dev) for v in (ops, off, x, t, k)]
    vals = torch.full((P, C), float("nan"), device=dev)
    fit = torch.full((P,), float("nan"), device=dev)
    flags = ctypes.c_uint32(0)
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(v.data_ptr()) for v in (*d, vals, fit)]
    rc = lib.gp_eval_small_noalloc(p[0], ctypes.c_size_t(ops.size), p[1], ctypes.c_uint32(P), p[2], p[3], p[4],
                                   ctypes.c_uint32(C), p[5], p[6], None, ctypes.byref(flags))
    assert rc == 0 and flags.value == 0
    ov, of = oracle.eval_pop_f32(tree, np.array([0, 1023], np.uint64), k, x, t)
    assert np.array_equal(oracle.canon_nan(vals.cpu().numpy()), np.repeat(oracle.canon_nan(ov), P, 0))
    assert np.array_equal(oracle.canon_nan(fit.cpu().numpy()), np.repeat(oracle.canon_nan(of), P, 0))
