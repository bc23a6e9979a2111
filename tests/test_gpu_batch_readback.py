"""Host read-back of a batch's moments: from several threads, and into page-locked memory."""
import ctypes as C
import threading

import numpy as np
import pytest

from paper_1411_6121_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(300, 171), (511, 257), (40, 21)]


@pytest.fixture(scope="module")
def batch():
    from paper_1411_6121_gb300 import dugks
    b = dugks.Batch([dict(shape=s, nu=0.05, bcs=W.cavity_bcs(2, 0.1)) for s in SHAPES], dt=0.5)
    for i, s in enumerate(SHAPES):
        b.init(i, *W.random_state_fields(s, seed=i + 1, u_amp=0.03, p_amp=1e-3))
    yield b, [b.moments(i) for i in range(len(SHAPES))]
    b.close()


def test_threads_read_instances_at_once(batch):
    b, want = batch
    wrong = []

    def read(i):
        for _ in range(60):
            if not np.array_equal(b.moments(i), want[i]):
                wrong.append(i)

    ts = [threading.Thread(target=read, args=(i,)) for i in range(len(SHAPES))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong, (len(wrong), sorted(set(wrong)))


def test_page_locked_destination(batch):
    import torch
    b, want = batch
    for i, (nx, ny) in enumerate(SHAPES):
        out = torch.zeros((3, nx * ny), dtype=torch.float32).pin_memory()
        b._check(b.lib.dugks_batch_moments(b.h, i, C.c_void_p(out.data_ptr()), 0))
        assert np.array_equal(out.numpy(), want[i])


def test_device_pointer_passed_as_host(batch):
    """The copy refuses it (or makes it, where the driver does): the host never writes through it."""
    import torch
    b, want = batch
    nx, ny = SHAPES[2]
    out = torch.zeros((3, nx * ny), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    rc = b.lib.dugks_batch_moments(b.h, 2, C.c_void_p(out.data_ptr()), 0)
    assert rc != 0 or np.array_equal(out.cpu().numpy(), want[2])
    assert np.array_equal(b.moments(2), want[2])
