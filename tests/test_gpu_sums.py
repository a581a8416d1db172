"""Rounding of the long sums, on the GPU, against the same sums in the shorter chains they may be split into.  The data are
such that every product is exact, so that the errors seen are those of the additions alone."""
import numpy as np
import pytest

from tests.gpu_common import dev_vec, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Solver():
    need_gpu()
    from paper_2506_18408_gb300 import Solver

    return Solver


def _bits(a, bits):
    m, e = np.frexp(a)
    return np.ldexp(np.round(m * 2.0 ** bits), e - bits)


def _lane_sums(p):
    """Row sums as 8 lanes (up to 64 entries) or 32 form them: every lane's entries in order, then a tree."""
    v = 8 if p.shape[1] <= 64 else 32
    lanes = []
    for j in range(v):
        s = np.zeros(p.shape[0], p.dtype)
        for i in range(j, p.shape[1], v):
            s = s + p[:, i]
        lanes.append(s)
    while len(lanes) > 1:
        h = len(lanes) // 2
        lanes = [lanes[j] + lanes[j + h] for j in range(h)]
    return lanes[0]


def _rms(e):
    return float(np.sqrt(np.mean(np.square(e.astype(np.float64)))))


# Rows that take a thread each, with a dominant entry anywhere in the row: no larger an error than the lanes' sums.  Emulated on
# the CPU, the ratio of the two is at most 1.05 (at 25 entries) and below 1 from 100 on; 16,383 rows give it to some 2 %.
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("length", [17, 25, 33, 64, 65, 100, 128, 256, 509, 512])
def test_long_rows_round_no_more_than_lanes(Solver, precision, length):
    n = 16384
    rng = np.random.default_rng(length)
    dt, bits = (np.float64, 26) if precision == "fp64" else (np.float32, 24)
    val = _bits(rng.standard_normal((n - 1, length)), bits)
    at = rng.integers(0, length, n - 1), np.arange(n - 1)
    val[at[1], at[0]] = 0.0
    val[at[1], at[0]] = _bits(1.2 * np.abs(val).sum(1), bits)
    col = rng.integers(0, n, (n - 1, length)).astype(np.int32)
    rp = np.concatenate([[0, 1], 1 + length * np.arange(1, n)]).astype(np.int64)
    sv = Solver(n, rp, np.concatenate([[3], col.ravel()]).astype(np.int32), np.concatenate([[1.0], val.ravel()]), sketch_seed=1,
                precision=precision, block_rows=8192)
    v = np.where(rng.random(n) < 0.5, -1.0, 1.0) / 128.0  # a unit vector
    _, k, _, B, _ = sv.inner_cycle(dev_vec(v), m=2, s=32, k=0)
    assert k == 2
    if precision == "fp64":
        x = _bits(rng.standard_normal(n), 26)
        got = sv.spmv(dev_vec(x)).cpu().numpy()
    else:  # the second basis vector without a window is A v, scaled; row 0 has one entry
        x, got = v, B[1].cpu().numpy()
        got = got * (v[3] / got[0])
    sv.close()
    p = val * x[col]
    exact = p.astype(np.longdouble).sum(1)
    assert np.array_equal(p.astype(dt).astype(np.float64), p)
    assert _rms(got[1:] - exact) <= 1.1 * _rms(_lane_sums(p.astype(dt)) - exact)


# The allocation-free sketch adds a vector's sums of 128 columns (short vectors) without the error of plain additions: no larger
# an error than that of sums that are exact over 1024 columns, whose own conversions and additions are two or three roundings.
@pytest.mark.parametrize("n,s,zeta", [(1500, 40, 4), (3000, 100, 4), (6000, 64, 1), (12_000, 100, 16), (32_000, 240, 8), (33_000, 240, 8)])
def test_allocation_free_sketch_of_short_vectors(n, s, zeta):
    need_gpu()
    from oracle import sketch as osk
    from paper_2506_18408_gb300 import sfgmres_sketch_apply_noalloc

    S = osk.sketch_matrix(n, s, zeta, 7)
    S.data = np.sign(S.data).astype(np.int64)
    S = S.astype(np.int64)
    got, plain = [], []
    for seed in range(8):
        q = np.round(np.clip(np.random.default_rng(seed).standard_normal(n), -3.9, 3.9) * 2.0 ** 50).astype(np.int64)
        c = dev_vec(np.full(s, np.nan))
        sfgmres_sketch_apply_noalloc(n, s, zeta, 7, dev_vec(q * 2.0 ** -50), c)
        blocks, edges = 0.0, range(0, n, 1024)
        for e in edges:
            blocks = blocks + (S[:, e:e + 1024] @ q[e:e + 1024]).astype(np.float64)
        exact = (S @ q).astype(np.longdouble)
        got.append(c.cpu().numpy().astype(np.longdouble) * (np.sqrt(zeta) * 2.0 ** 50) - exact)
        plain.append(blocks - exact)
    assert _rms(np.array(got)) <= 1.05 * _rms(np.array(plain))
