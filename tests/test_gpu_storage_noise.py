"""The stochastic rounding of 16-bit stores draws each value's random bits from the step, the cell and
the velocity alone, so that a run's noise is the same whichever kernel makes the step.

One step of the default kernel against the reference kernel (kernel=1) from the same stored state. The
two differ by FP32 rounding (some 2e-7 of the largest value), which turns the rounding of a value v of
p significant bits with a probability of about 2e-7 max|v| / (2^-p |v|): a few in a thousand. Other random
bits would turn it with probability 2 f (1 - f), f the discarded fraction: a third of all values."""
import numpy as np
import pytest

from paper_1411_6121_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "2d_odd": dict(shape=(61, 37), q=9, bcs=W.cavity_bcs(2, 0.1)),
    "2d_tall": dict(shape=(40, 300), q=9, bcs=W.cavity_bcs(2, 0.1)),
    "2d_forced": dict(shape=(128, 33), q=9, bcs=W.channel_bcs(2), g=(1e-4, -2e-5, 0.0)),
    "d3q27": dict(shape=(35, 13, 9), q=27, bcs=W.cavity_bcs(3, 0.1)),
    "d3q27_forced": dict(shape=(31, 14, 6), q=27, bcs=W.channel_bcs(3), g=(1e-4, -2e-5, 3e-5)),
}


@pytest.mark.parametrize("store", [1, 2])
@pytest.mark.parametrize("name", sorted(CASES))
def test_noise_does_not_depend_on_the_kernel(name, store):
    from paper_1411_6121_gb300 import dugks
    cfg = dict(nu=0.05, dt=0.5, store=store, **CASES[name])
    p, u = W.random_state_fields(cfg["shape"], seed=11, u_amp=0.03, p_amp=1e-3)
    outs = []
    for kernel in (0, 1):
        s = dugks.Sim(kernel=kernel, **cfg)
        s.init(p=p, u=u)
        s.step(1)
        outs.append(np.asarray(s.get_state(), dtype=np.float64))
        s.close()
    assert np.mean(outs[0] != outs[1]) < 0.05
