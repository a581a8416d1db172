"""What a handle's earlier calls must not change: results and the set-up a call needs, on the GPU."""
import numpy as np
import pytest

from tests.gpu_common import dev_vec, need_gpu

import workloads

pytestmark = pytest.mark.gpu
PAR = dict(m=30, s=120, k=2, tol=1e-8)


@pytest.fixture(scope="module")
def Solver():
    need_gpu()
    from paper_2506_18408_gb300 import Solver

    return Solver


# y = A x with rows of 0 to 700 entries, one thread, 8 lanes or a warp each: the same bits on a fresh handle, after solves, and
# after new values while the blocks of many right-hand sides are current
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_product_does_not_depend_on_earlier_calls(Solver, precision):
    n = 9000
    rng = np.random.default_rng(5)
    length = rng.choice(np.asarray([0, 3, 15, 16, 30, 64, 65, 200, 513, 700]), n)
    rp = np.concatenate([[0], np.cumsum(length + 1)]).astype(np.int64)
    rows = np.repeat(np.arange(n), length + 1)
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    col[rp[:-1]] = np.arange(n)
    val = rng.standard_normal(rp[-1])
    val[rp[:-1]] = 2.0 * (np.bincount(rows, np.abs(val), n) + np.bincount(col, np.abs(val), n))
    x, many = dev_vec(rng.standard_normal(n)), dev_vec(rng.standard_normal(7 * n))
    new = val * np.linspace(1.0, 1.5, len(val))

    def fresh(v):
        sv = Solver(n, rp, col, v, sketch_seed=1, precision=precision)
        y = sv.spmv(x).cpu().numpy()
        sv.close()
        return y

    sv = Solver(n, rp, col, val, sketch_seed=1, precision=precision)
    want = fresh(val)
    assert np.array_equal(sv.spmv(x).cpu().numpy(), want)
    sv.solve(x, **PAR)
    assert np.array_equal(sv.spmv(x).cpu().numpy(), want)
    sv.solve_batch(many, nrhs=7, **PAR)
    sv.update_values(dev_vec(new))
    assert np.array_equal(sv.spmv(x).cpu().numpy(), fresh(new))
    sv.solve(x, transpose=True, **PAR)
    sv.update_values(dev_vec(val))
    sv.solve_batch(many, nrhs=7, transpose=True, **PAR)
    assert np.array_equal(sv.spmv(x).cpu().numpy(), want)
    sv.close()
