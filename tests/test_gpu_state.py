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


# Single solves, several numbers of right-hand sides (row blocks of as many sizes), y = A x and S v in turn: what each needs is
# built once, so that later rounds launch only the solves' own kernels, and give the same bits.
@pytest.mark.parametrize("kind", ["convdiff", "zipf"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_calls_in_turn_build_their_row_blocks_once(Solver, kind, precision):
    A = workloads.convdiff(64, (30.0, 10.0)) if kind == "convdiff" else workloads.random_zipf(6000, seed=3)
    sv = Solver(A.n, A.row_ptr, A.col, A.val, sketch_seed=1, precision=precision)
    counts = (1, 2, 4, 8, 16)
    b = {r: dev_vec(workloads.rhs(r * A.n, seed=r)) for r in counts}
    rounds = []
    for _ in range(4):
        launches, out = [], []
        for r in counts:
            x, info = sv.solve(b[1], **PAR) if r == 1 else sv.solve_batch(b[r], nrhs=r, **PAR)
            assert info["status"] == 0
            launches.append(info["kernel_launches"])
            out += [x.cpu().numpy(), sv.spmv(b[1]).cpu().numpy(), sv.sketch(b[1], 120).cpu().numpy()]
        rounds.append((launches, out))
    for launches, out in rounds[1:]:
        assert all(q < p for q, p in zip(launches[1:], rounds[0][0][1:])) and launches == rounds[1][0]
        assert all(np.array_equal(p, q) for p, q in zip(out, rounds[0][1]))
    sv.close()


# a captured outer step is not replayed on row blocks built anew: sizes set back and forth with cycles, products and sketches (which
# capture nothing) between two solves, more sizes than a handle keeps
@pytest.mark.parametrize("kind", ["convdiff", "zipf"])
def test_replay_after_row_blocks_were_rebuilt(Solver, kind):
    A = workloads.convdiff(64, (30.0, 10.0)) if kind == "convdiff" else workloads.random_zipf(6000, seed=3)
    sv = Solver(A.n, A.row_ptr, A.col, A.val, sketch_seed=1, block_rows=512)
    b = dev_vec(workloads.rhs(A.n, seed=0))
    v = b / b.norm()
    want = sv.solve(b, **PAR)[0].cpu().numpy()
    for rows in range(544, 544 + 32 * 40, 32):
        sv.set("block_rows", rows)
        sv.inner_cycle(v, m=4, s=120, k=2)
        sv.spmv(b)
    sv.set("block_rows", 512)
    assert np.array_equal(sv.solve(b, **PAR)[0].cpu().numpy(), want)
    sv.autotune(m=30, s=120, k=2)
    sv.set("block_rows", 512)
    sv.set("spmv_vector", 0)
    assert np.array_equal(sv.solve(b, **PAR)[0].cpu().numpy(), want)
    sv.close()


# Blocks of several waves, where every step is two launches: the QR staged in shared memory (it waits for an SM) and, beside the
# steps the caller asks to split, read from L2 form the same sums, in cycles and solves.
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_blocks_of_several_waves(Solver, precision):
    A = workloads.convdiff(150, (30.0, 10.0))
    b = dev_vec(workloads.rhs(A.n, seed=4))
    sv = Solver(A.n, A.row_ptr, A.col, A.val, sketch_seed=1, precision=precision, block_rows=32)
    got = []
    for fused in (1, 0):
        sv.set("fused_step", fused)
        z = sv.inner_cycle(b / b.norm(), m=100, s=400, k=2)[0].cpu().numpy()
        x, info = sv.solve(b, m=100, s=400, k=2, tol=1e-8)
        r = A.to_scipy() @ x.cpu().numpy() - b.cpu().numpy()
        assert info["status"] == 0 and np.linalg.norm(r) <= 1.01e-8 * float(b.norm())
        got.append((z, x.cpu().numpy()))
    assert all(np.array_equal(p, q) for p, q in zip(*got))
    sv.close()
