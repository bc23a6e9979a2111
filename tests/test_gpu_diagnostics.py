"""Precision of the residual and the totals: FP64 in u, its difference, the squares and the sums, over cell
sums of 32- and 16-bit states that hold 2^-47 of sum |g|."""
import ctypes as C

import numpy as np
import pytest

from paper_1411_6121_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RT = 0.4  # c = sqrt(1.2): the velocities fill an FP64 significand


def _e(q):
    d = 2 if q == 9 else 3
    e = np.stack(np.meshgrid(*[[-1.0, 0.0, 1.0]] * d, indexing="ij")).reshape(d, -1)
    return e[:, np.abs(e).sum(0) < 3] if q == 19 else e


def _static(q, shape, state, uprev, have_prev):
    import torch
    from paper_1411_6121_gb300 import dugks
    lib = dugks.load()
    n3 = tuple(shape) + (1,) * (3 - len(shape))
    out = np.zeros(len(shape) + 2)
    st = torch.tensor(state, device="cuda")
    up = torch.tensor(uprev, device="cuda")
    torch.cuda.synchronize()
    rc = lib.dugks_residual_static(q, 0, C.c_void_p(st.data_ptr()), *n3, RT, 1.0, None, None, C.c_void_p(up.data_ptr()),
                                   have_prev, out.ctypes.data_as(C.POINTER(C.c_double)), None)
    assert rc == 0
    return out, up.cpu().numpy()


@pytest.mark.parametrize("shape", [(6, 4), (7, 5)])
def test_cell_sums_of_cancelling_values(shape):
    """Large values of two pairs that cancel along x and leave a small one: every cell alike, so that what is
    lost adds up. The error of a cell's sums is at most 2^-47 sum |g|, that of the totals the cells' sum of
    it (and FP64 rounding, far below)."""
    from paper_1411_6121_gb300 import dugks
    n = int(np.prod(shape))
    e = _e(9)
    k = {tuple(v): i for i, v in enumerate(e.T.astype(int))}
    big, small = np.float32(0.3), np.float32(0.7 * 2.0 ** -30)
    g = np.zeros((9, n), np.float32)
    g[k[1, 1]], g[k[1, -1]], g[k[1, 0]] = big, -big, small
    s = dugks.Sim(shape, q=9, nu=0.05, dt=0.5, rt=RT, bcs=W.all_periodic())
    s.set_state(g)
    r = s.residual()
    s.close()
    c = np.sqrt(3 * RT)
    want = c * n * (e @ g[:, 0].astype(np.float64))
    bound = c * n * 2.0 ** -47 * float(np.abs(g[:, 0].astype(np.float64)).sum())
    assert np.abs(r[2:] - want).max() <= bound, (r[2:] - want, bound)
    assert abs(r[1] - n * (1.0 + float(g[:, 0].astype(np.float64).sum()))) <= bound / c + n * 2.0 ** -52


@pytest.mark.parametrize("q,shape", [(9, (30, 14)), (19, (13, 7, 5)), (27, (8, 6, 5))])
def test_previous_velocity_is_read_and_kept_in_fp64(q, shape):
    """State values of few bits, whose sums are exact: u = c j is one FP64 product, the velocity handed back
    is within an ulp of it, and a velocity that differs by 2^-48 is seen to differ by that (two FP64
    roundings of 2^-53 on it: 2^-4; a tenth allowed)."""
    rng = np.random.default_rng(q)
    n = int(np.prod(shape))
    g = (rng.integers(-(1 << 11), 1 << 11, size=(q, n)) / 2.0 ** 15).astype(np.float32)
    u = np.sqrt(3 * RT) * (_e(q) @ g.astype(np.float64))
    out, up = _static(q, shape, g, u * (1 + 2.0 ** -48), 1)
    assert np.all(np.abs(up - u) <= 2.0 ** -52 * np.abs(u))
    assert abs(out[0] * 2.0 ** 48 - 1) < 0.1, out[0] * 2.0 ** 48


def test_small_and_large_velocities():
    """The squares keep the range of FP64: a decayed flow, and one that has blown up but is finite."""
    rng = np.random.default_rng(1)
    for scale in (1e-33, 1e15):
        g = (scale * rng.standard_normal((9, 42))).astype(np.float32)
        before = (scale * rng.standard_normal((9, 42))).astype(np.float32)
        u, v = (np.sqrt(3 * RT) * (_e(9) @ x.astype(np.float64)) for x in (g, before))
        out, _ = _static(9, (6, 7), g, v, 1)
        want = np.linalg.norm((u - v) / scale) / np.linalg.norm(u / scale)
        assert abs(out[0] / want - 1) < 1e-12, (scale, out[0], want)
