"""Kernels at the edges of their tiles, on the GPU: lengths around the pieces a CTA or a warp takes, remainders of their
unrolled loops, the smallest and largest sizes, against NumPy arithmetic on the same values."""
import os
import subprocess
import sys

import numpy as np
import pytest

from tests.gpu_common import dev_vec, need_gpu

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Solver():
    need_gpu()
    from paper_2506_18408_gb300 import Solver

    return Solver


def _unit(n, seed):
    v = np.random.default_rng(seed).standard_normal(n)
    return dev_vec(v / np.linalg.norm(v))


# z = B y: pieces of 512 (FP64) or 1024 (FP32, BF16) rows of a block, four columns at a time
@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("n,m,block_rows", [(33, 1, 0), (511, 3, 512), (512, 4, 512), (513, 5, 512), (1025, 7, 8192),
                                            (3 * 1024 + 1, 9, 1056), (8191, 34, 8192)])
def test_correction_is_the_basis_times_y(Solver, precision, n, m, block_rows):
    A = workloads.convdiff(n, (30.0,))
    sv = Solver(A.n, A.row_ptr, A.col, A.val, sketch_seed=1, precision=precision, block_rows=block_rows)
    z, k, _, B, y = sv.inner_cycle(_unit(n, n), m=m, s=max(32, 4 * m) if n > 256 else 32, k=2)
    B, y, z = B[:k].cpu().numpy(), y.cpu().numpy(), z.cpu().numpy()
    size = np.abs(y) @ np.abs(B)
    # FP64: k products and sums, the coefficients' and the exported basis's own roundings.  FP32 pairs: two-term
    # coefficients (2^-47 each) and a low part whose k sums each round to 2^-24 of at most k 2^-23 of the whole.
    bound = (2 * k + 8) * 2.0 ** -53 if precision == "fp64" else (k + 8) ** 2 * 2.0 ** -46
    assert np.all(np.abs(z - y @ B) <= bound * size + 1e-300)
    sv.close()


# the sketched QR: fewer sketch rows than CTAs of its cluster, rows just past a warp, more columns than threads, slices that
# do not fit in shared memory; clusters of 2, 4 and 16 CTAs
@pytest.mark.parametrize("N,m,s", [(20, 8, 8), (30, 24, 33), (40, 40, 160), (60, 130, 520), (70, 300, 1000), (70, 600, 1200)])
def test_sketched_least_squares_is_optimal(Solver, N, m, s):
    from oracle import sketch as osk

    A = workloads.convdiff(N, (30.0, 10.0))
    sv = Solver(A.n, A.row_ptr, A.col, A.val, sketch_seed=1)
    v = _unit(A.n, m)
    _, k, _, B, y = sv.inner_cycle(v, m=m, s=s, k=2)
    assert k > min(m, 100) // 2
    S = osk.sketch_matrix(A.n, s, 8, 1)
    C = S @ (A.to_scipy() @ B[:k].cpu().numpy().T)
    c, y = S @ v.cpu().numpy(), y.cpu().numpy()
    # Gram-Schmidt with reorthogonalisation solves a problem perturbed by O(k s u) relative to its data
    size = np.linalg.norm(C) * (np.linalg.norm(c) + np.linalg.norm(C) * np.linalg.norm(y))
    assert np.linalg.norm(C.T @ (c - C @ y)) <= 8 * k * s * 2.0 ** -53 * size
    sv.close()


# row blocks whose shared memory is just under the 48 KB a launch gets by default, in a process that has not raised it yet
@pytest.mark.parametrize("block_rows", [5632, 6112, 6144])
def test_blocks_just_under_the_default_shared_memory(Solver, block_rows):
    code = f"""
import sys; sys.path.insert(0, '.')
import torch, workloads
from paper_2506_18408_gb300 import Solver
A = workloads.convdiff(90, (30.0, 10.0))
b = torch.from_numpy(workloads.rhs(A.n, seed=0)).cuda()
x, info = Solver(A.n, A.row_ptr, A.col, A.val, block_rows={block_rows}).solve(b, m=30, s=120, k=2, tol=1e-8)
sys.exit(info['status'])
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    assert subprocess.run([sys.executable, "-c", code], cwd=root).returncode == 0


# single and many right-hand sides use row blocks of different sizes on one handle: alternating between them, with new values
# in between, gives what fresh handles give, bit for bit
@pytest.mark.parametrize("kind", ["convdiff", "zipf"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_alternating_numbers_of_right_hand_sides(Solver, kind, precision):
    A = workloads.convdiff(40, (30.0, 10.0)) if kind == "convdiff" else workloads.random_zipf(6000, seed=3)
    par = dict(m=30, s=120, k=2, tol=1e-8)
    one, many = dev_vec(workloads.rhs(A.n, seed=0)), dev_vec(workloads.rhs(7 * A.n, seed=1))
    vals = [dev_vec(A.val), dev_vec(A.val * np.linspace(1.0, 1.5, A.nnz))]

    def call(sv, nrhs):
        return (sv.solve(one, **par) if nrhs == 1 else sv.solve_batch(many, nrhs=nrhs, **par))[0].cpu().numpy()

    sv = Solver(A.n, A.row_ptr, A.col, A.val, sketch_seed=1, precision=precision)
    for which, nrhs in ((0, 1), (0, 7), (0, 1), (1, 1), (1, 7), (0, 7), (1, 1)):
        sv.update_values(vals[which])
        fresh = Solver(A.n, A.row_ptr, A.col, vals[which].cpu().numpy(), sketch_seed=1, precision=precision)
        assert np.array_equal(call(sv, nrhs), call(fresh, nrhs))
        fresh.close()
    sv.close()


# FP32 inner cycles: the staged SpMV with rows of 0 to 16 entries in every order, row groups cut by the block's and the
# system's end, entries that start anywhere within 16 bytes
@pytest.mark.parametrize("n,maxlen,block_rows", [(31, 1, 32), (33, 16, 32), (1000, 5, 512), (5000, 9, 544), (4097, 16, 1024),
                                                 (20_000, 3, 8192)])
def test_staged_spmv_with_ragged_rows(Solver, n, maxlen, block_rows):
    rng = np.random.default_rng(n + maxlen)
    length = rng.integers(0, maxlen + 1, n)
    length[0], length[n // 2] = maxlen, 0
    rp = np.concatenate([[0], np.cumsum(length)]).astype(np.int64)
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    val = rng.standard_normal(rp[-1])
    sv = Solver(n, rp, col, val, sketch_seed=1, precision="fp32", block_rows=block_rows)
    v = _unit(n, 1)
    # the second basis vector is A b_1 minus its projection on b_1, normalised
    _, k, _, B, _ = sv.inner_cycle(v, m=2, s=16, k=1)
    b1 = B[0].cpu().numpy()
    A = np.zeros(n)
    np.add.at(A, np.repeat(np.arange(n), length), val.astype(np.float32).astype(np.float64) * b1[col])
    w = A - b1 * (b1 @ A)
    w /= np.linalg.norm(w)
    got = B[1].cpu().numpy()
    # FP32: maxlen products and sums per row, the projection's and the scale's roundings, the dot's over n rows
    assert k == 2 and np.linalg.norm(got - w) <= (maxlen + 8 + np.sqrt(n)) * 2.0 ** -24 * max(1.0, np.linalg.norm(A) / np.linalg.norm(A - b1 * (b1 @ A)))
    sv.close()


# the allocation-free sketch: vectors around one chunk of columns and one wave of CTAs, counts of nonzeros with and without a
# compile-time kernel, values of very different size
@pytest.mark.parametrize("n,s,zeta", [(1, 1, 1), (127, 16, 2), (129, 40, 3), (992, 33, 4), (38_913, 100, 16), (301_568, 240, 8),
                                      (301_569, 31, 5)])
def test_allocation_free_sketch_at_chunk_edges(Solver, n, s, zeta):
    from oracle import sketch as osk
    from paper_2506_18408_gb300 import sfgmres_sketch_apply_noalloc

    rng = np.random.default_rng(n)
    v = rng.standard_normal(n) * 10.0 ** rng.integers(-3, 4, n)
    c = dev_vec(np.full(s, np.nan))
    d = dev_vec(v)
    sfgmres_sketch_apply_noalloc(n, s, zeta, 7, d, c)  # the default stream, as c's copy below
    S = osk.sketch_matrix(n, s, zeta, 7)
    count = np.asarray(abs(S).sign().sum(axis=1)).ravel()
    # both sides: a rounding per term and per addition (of the chunk's largest value, or of the running sum)
    bound = 2.0 ** -53 * ((2 * count + n / 128 + 8) * (abs(S) @ np.abs(v)) + count * np.abs(v).max())
    assert np.all(np.abs(c.cpu().numpy() - S @ v) <= bound)


# y = A x and full solves through the outer kernels' staged SpMV: pieces of 2048 rows, rows of 0 to 16 entries, blocks too
# large for the stage area beside them
@pytest.mark.parametrize("n,maxlen,block_rows", [(1, 1, 0), (33, 16, 32), (2049, 7, 8192), (9000, 16, 4128), (20_000, 9, 8192)])
def test_staged_fp64_spmv(Solver, n, maxlen, block_rows):
    rng = np.random.default_rng(n + maxlen)
    length = rng.integers(0, maxlen, n)
    rp = np.concatenate([[0], np.cumsum(length + 1)]).astype(np.int64)
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    val = rng.standard_normal(rp[-1])
    col[rp[:-1]] = np.arange(n)
    val[rp[:-1]] = 8.0 * maxlen
    sv = Solver(n, rp, col, val, sketch_seed=1, block_rows=block_rows, zeta=min(8, n))
    x = rng.standard_normal(n)
    y, size = np.zeros(n), np.zeros(n)
    rows = np.repeat(np.arange(n), length + 1)
    np.add.at(y, rows, val * x[col])
    np.add.at(size, rows, np.abs(val * x[col]))
    assert np.all(np.abs(sv.spmv(dev_vec(x)).cpu().numpy() - y) <= 2 * (maxlen + 1) * 2.0 ** -53 * size)
    if n > 64:
        got, info = sv.solve(dev_vec(y), m=20, s=80, k=2, tol=1e-10)
        r = y.copy()
        np.subtract.at(r, rows, val * got.cpu().numpy()[col])
        assert info["status"] == 0 and abs(info["rel_res_true"] - np.linalg.norm(r) / np.linalg.norm(y)) <= 1e-14
    sv.close()


# the length-binned SpMV before and after the sorted copy exists: empty rows, rows beyond the copy's longest, blocks whose long
# rows the copy leaves out, slices cut by a block's end, new values, FP64 and FP32 cycles on one handle, the transpose
@pytest.mark.parametrize("n,lens,block_rows", [(70, (0, 70), 32), (3000, (0, 3, 17, 64, 65, 513, 700), 512), (3000, (17,), 1024),
                                               (9001, (1, 4, 4, 4, 5, 30, 200), 0), (20_000, (4, 4, 4, 40, 256), 8192)])
def test_length_binned_spmv_classes(Solver, n, lens, block_rows):
    rng = np.random.default_rng(n + len(lens))
    length = rng.choice(np.asarray(lens), n)
    rp = np.concatenate([[0], np.cumsum(length + 1)]).astype(np.int64)
    rows = np.repeat(np.arange(n), length + 1)
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    col[rp[:-1]] = np.arange(n)
    x = rng.standard_normal(n)
    sv = None
    for scale in (1.0, 3.0):
        val = scale * rng.standard_normal(rp[-1])
        val[rp[:-1]] = scale * 2.0 * (np.bincount(rows, np.abs(val), n) + np.bincount(col, np.abs(val), n))
        if sv is None:
            sv = Solver(n, rp, col, val, sketch_seed=1, block_rows=block_rows)
        else:
            sv.update_values(dev_vec(val))
        y, size = np.bincount(rows, val * x[col], n), np.bincount(rows, np.abs(val * x[col]), n)
        for precision in ("fp64", "fp32"):
            sv.set("precision", precision)
            for transpose in (False, True):
                b = np.bincount(col, val * x[rows], n) if transpose else y
                got, info = sv.solve(dev_vec(b), m=12, s=48, k=2, tol=1e-12, transpose=transpose)
                assert info["status"] == 0 and np.linalg.norm(got.cpu().numpy() - x) <= 1e-10 * np.linalg.norm(x)
            err = np.abs(sv.spmv(dev_vec(x)).cpu().numpy() - y)
            assert np.all(err <= (length + 8) * 2.0 ** -53 * 2 * size)
    sv.close()


# the sketch sums' pieces: the step of one launch (11 to 14 warps sum lists) and of two (16 warps) form the same sums, bit for
# bit, also in FP32, for one group of sketch rows up to more groups than warps
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("s,t", [(24, 0), (70, 1), (130, 2), (160, 2), (224, 3), (256, 4), (352, 4), (400, 2), (520, 2)])
def test_sketch_pieces_do_not_depend_on_the_launches(Solver, precision, s, t):
    A = workloads.convdiff(150, (30.0, 10.0))
    v = _unit(A.n, s)
    sv = Solver(A.n, A.row_ptr, A.col, A.val, sketch_seed=1, precision=precision)
    got = []
    for fused in (1, 0):
        sv.set("fused_step", fused)
        got.append(sv.inner_cycle(v, m=8, s=s, k=t)[0].cpu().numpy())
    assert np.array_equal(*got)
    sv.close()


# ILU(0) passes multiply by the pivots' reciprocals, or divide where one overflows, also after new values between replays.  z =
# y_0 M^{-1} v by the two colours' substitutions; where v is zero the scale of the row cancels.  Bound: eight roundings of
# products and sums beside 1e-310 (units of 2^-1074, some 4e-13 of the pivot), and FP64's own.
@pytest.mark.parametrize("n", [64, 513, 1025])
def test_ilu_pivot_without_a_reciprocal(Solver, n):
    A = workloads.convdiff(n, (5.0,))
    val, k = A.val / abs(A.val).max(), 33
    v = np.random.default_rng(n).standard_normal(n)
    v[k] = 0.0
    v /= np.linalg.norm(v)
    M = A.to_scipy().tocsr()
    M.data = val.copy()
    odd, even = np.arange(1, n, 2), np.arange(0, n, 2)
    d = M.diagonal()
    L, U = M[odd][:, even] @ np.diag(1.0 / d[even]), M[even][:, odd].toarray()
    want = np.empty(n)
    want[odd] = (v[odd] - L @ v[even]) / (d[odd] - np.einsum("ij,ji->i", L, U))
    want[even] = (v[even] - U @ want[odd]) / d[even]
    small = val.copy()
    small[A.row_ptr[k]:A.row_ptr[k + 1]] *= 1e-310
    sv = Solver(n, A.row_ptr, A.col, val, sketch_seed=1, precond=1, max_outer=200)
    for values in (val, small, val):
        sv.update_values(dev_vec(values))
        z, kk, _, _, y = sv.inner_cycle(dev_vec(v), m=1, s=32, k=1)
        z, y = z.cpu().numpy(), float(y.cpu()[0])
        assert kk == 1 and y != 0.0
        assert np.max(np.abs(z / y - want)) <= 1e-12 + 1e-14 * np.max(np.abs(want))
        x, info = sv.solve(dev_vec(v), m=30, s=60, k=2, tol=1e-8)
        M.data = values.copy()
        assert info["status"] == 0 and np.linalg.norm(v - M @ x.cpu().numpy()) <= 1.01e-8
    sv.close()
