"""The step kernels at the edges of their tiles, element by element against the oracle: sizes one
below, at and one above the columns and rows of a tile, odd sizes (the last column alone in its
lane), every wall type on both axes, with and without a force; and the same bits whatever the
block's rows (2D)."""
import numpy as np
import pytest

from oracle import Oracle
from paper_1411_6121_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FLOWS = {
    "channel": dict(bcs=W.channel_bcs(2), g=(1e-4, -2e-5, 0.0)),
    "cavity": dict(bcs=W.cavity_bcs(2, 0.1)),
    "box": dict(bcs=[W.pressure(1e-3), W.wall((0.0, 0.02)), W.bounce_back((0.03, 0.0)), W.bounce_back()], g=(0.0, 1e-4, 0.0)),
    "periodic": dict(bcs=W.all_periodic()),
}
SIZES = [(2, 2), (3, 5), (59, 6), (60, 7), (61, 13), (62, 2), (121, 3)]


def _state(o):
    _, Wt = o.lattice()
    return o.get_state() - Wt[:, None] * o.cfg.rho0


def _pair(cfg, steps, **kw):
    from paper_1411_6121_gb300 import dugks
    p, u = W.random_state_fields(cfg["shape"], seed=sum(cfg["shape"]), u_amp=0.03, p_amp=1e-3)
    o = Oracle(**cfg)
    o.init(p=p, u=u)
    o.step(steps)
    s = dugks.Sim(**cfg, **kw)
    s.init(p=p, u=u)
    s.step(steps)
    return _state(o), s.get_state().astype(np.float64)


@pytest.mark.parametrize("flow", sorted(FLOWS))
@pytest.mark.parametrize("shape", SIZES)
def test_d2q9_tile_edges(shape, flow):
    cfg = dict(shape=shape, q=9, nu=0.05, dt=0.5, **FLOWS[flow])
    ref, got = _pair(cfg, 10)
    assert np.abs(got - ref).max() < 2e-6 * np.abs(ref).max()


@pytest.mark.parametrize("flow", sorted(FLOWS))
@pytest.mark.parametrize("shape", [(9, 724), (31, 604), (78, 883), (1140, 49)])
def test_d2q9_either_side_of_the_one_cell_rule(shape, flow):
    """Meshes that the one-cell kernel takes (the first three) and one beyond its rule."""
    cfg = dict(shape=shape, q=9, nu=0.05, dt=0.5, **FLOWS[flow])
    ref, got = _pair(cfg, 10)
    assert np.abs(got - ref).max() < 2e-6 * np.abs(ref).max()


@pytest.mark.parametrize("flow", ["box", "channel"])
def test_d2q9_bits_do_not_depend_on_the_block(flow):
    cfg = dict(shape=(67, 31), q=9, nu=0.05, dt=0.5, **FLOWS[flow])
    outs = [_pair(cfg, 8, **kw)[1] for kw in ({}, dict(tile=(32, 4)), dict(tile=(32, 8)), dict(tile=(32, 16)))]
    for o in outs[1:]:
        assert np.array_equal(o, outs[0])


@pytest.mark.parametrize("shape", [(61, 7), (9, 33)])
def test_d2q9_f16_one_step(shape):
    """One step from the same stored state: within one stored rounding (2^-10) of the FP64 step."""
    from paper_1411_6121_gb300 import dugks
    cfg = dict(shape=shape, q=9, nu=0.05, dt=0.5, **FLOWS["box"])
    p, u = W.random_state_fields(shape, seed=3, u_amp=0.03, p_amp=1e-3)
    s = dugks.Sim(store=2, **cfg)
    s.init(p=p, u=u)
    g0 = s.get_state().astype(np.float64) / 4096.0
    o = Oracle(**cfg)
    _, Wt = o.lattice()
    o.set_state(g0 + Wt[:, None] * o.cfg.rho0)
    o.step(1)
    s.step(1)
    ref, got = _state(o), s.get_state().astype(np.float64) / 4096.0
    assert np.all(np.abs(got - ref) <= 2e-6 * np.abs(ref).max() + 2.0 ** -10 * np.abs(ref))


FLOWS_3D = {
    "channel": dict(bcs=W.channel_bcs(3), g=(1e-4, -2e-5, 3e-5), omega=0.2),
    "cavity": dict(bcs=W.cavity_bcs(3, 0.1)),
    "box": dict(bcs=[W.pressure(1e-3), W.bounce_back((0.0, 0.02, 0.0)), W.bounce_back(), W.wall((0.03, 0.0, 0.0)),
                     W.wall(), W.bounce_back()], g=(0.0, 1e-4, 0.0)),
}


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("flow", sorted(FLOWS_3D))
@pytest.mark.parametrize("shape", [(29, 5, 2), (30, 6, 9), (31, 7, 17), (61, 13, 3)])
def test_3d_tile_edges(shape, flow, q):
    cfg = dict(shape=shape, q=q, nu=0.05, dt=0.5, **FLOWS_3D[flow])
    ref, got = _pair(cfg, 6)
    assert np.abs(got - ref).max() < 2e-6 * np.abs(ref).max()


# The kernel of FP64 storage and of non-uniform meshes: tiles of 30 columns and up to 6 rows. The
# tolerances are those of a step's rounding in either type (as in the parity tests), for 10 steps.
@pytest.mark.parametrize("flow", sorted(FLOWS))
@pytest.mark.parametrize("shape", [(2, 2), (29, 7), (30, 6), (31, 13), (61, 5)])
@pytest.mark.parametrize("mesh,store", [("uniform", 3), ("tanh", 3), ("tanh", 0)])
def test_d2q9_lean_tile_edges(mesh, store, shape, flow):
    cfg = dict(shape=shape, q=9, nu=0.05, dt=0.5, **FLOWS[flow])
    if mesh == "tanh":
        faces = [W.tanh_faces(n, n) for n in shape]
        cfg.update(faces=faces, dt=0.5 * min(np.diff(f).min() for f in faces))
    ref, got = _pair(cfg, 10, store=store)
    assert np.abs(got - ref).max() < (1e-11 if store == 3 else 2e-6) * np.abs(ref).max()


def test_d2q9_lean_matches_reference_kernel_with_field():
    """The default route of FP64 against the general kernel (kernel=1): a field, an oscillating
    acceleration, both orders of the walls."""
    import torch
    from paper_1411_6121_gb300 import dugks
    shape = (43, 19)
    fld = torch.tensor(W.force_field(shape, 2e-5, seed=2, rel=0.5), dtype=torch.float32, device="cuda")
    for bcs in (W.channel_bcs(2), W.channel_bcs(2)[2:] + W.channel_bcs(2)[:2]):
        outs = []
        for kernel in (0, 1):
            s = dugks.Sim(shape, q=9, nu=0.05, dt=0.5, g=(1e-5, 2e-5, 0.0), omega=0.3, bcs=bcs, field=fld, store=3, kernel=kernel)
            s.init(*W.random_state_fields(shape, seed=4, u_amp=0.03, p_amp=1e-3))
            s.step(10)
            outs.append(s.get_state())
        assert np.abs(outs[0] - outs[1]).max() < 1e-11 * np.abs(outs[1]).max()


@pytest.mark.parametrize("shapes", [[(2, 2), (300, 171)], [(511, 257), (7, 5)]])
def test_batch_read_back_by_pieces(shapes):
    """Moments read to the host by page-locked pieces: instances below, and of several (odd) pieces;
    the same values as the moments of the single instance."""
    from paper_1411_6121_gb300 import dugks
    ins = [dict(shape=s, nu=0.05, bcs=W.cavity_bcs(2, 0.1)) for s in shapes]
    b = dugks.Batch(ins, dt=0.5)
    for i, s in enumerate(shapes):
        p, u = W.random_state_fields(s, seed=7, u_amp=0.03, p_amp=1e-3)
        b.init(i, p=p, u=u)
        one = dugks.Sim(q=9, dt=0.5, tile=(32, 8), kernel=0, **ins[i])
        one.init(p=p, u=u)
        assert np.array_equal(b.moments(i), one.moments())
        one.close()
    b.close()


@pytest.mark.parametrize("shape", [(2, 400001), (1970000, 2)])
def test_d2q9_lean_long_meshes(shape):
    """FP64 meshes longer than a grid's y extent of tiles, along either axis: the general kernel's step."""
    from paper_1411_6121_gb300 import dugks
    p, u = W.random_state_fields(shape, seed=5, u_amp=0.03, p_amp=1e-3)
    outs = []
    for kernel in (0, 1):
        s = dugks.Sim(shape, q=9, nu=0.05, dt=0.5, bcs=W.all_periodic(), store=3, kernel=kernel)
        s.init(p=p, u=u)
        s.step(2)
        outs.append(s.get_state())
        s.close()
    assert np.abs(outs[0] - outs[1]).max() < 1e-11 * np.abs(outs[1]).max()
