"""A wait for the tensor cores that runs out in the middle of an epoch: the
weights, Adam's moments and its step count stay those of the steps before."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
N, BATCH, LR, SEED = 56, 16, 1e-3, 0x5EED  # the last batch is short


@pytest.mark.parametrize("step", [0, 2, 3])
def test_training_stops_at_the_failing_step(step):
    import paper_1708_08434_gb300 as p
    rng = np.random.default_rng(4)
    w = synth.cnn_initial_params().astype(np.float32)
    x = rng.uniform(-1.0, 1.0, (N, 1000, 2)).astype(np.float32)
    t = 0.3 * rng.standard_normal((N, 512)).astype(np.float32)
    a, b = p.Network(N, N), p.Network(N, N)
    for net in (a, b):
        net.set_params(w)
    a.load_samples(x, t)
    a.wait_selftest(step)
    with pytest.raises(p.SmError) as e:
        a.train(1, BATCH, LR, SEED)
    assert e.value.code == p.SM_ETIMEOUT
    order = np.argsort([int(synth.splitmix64(SEED ^ i, np.zeros(1))[0]) for i in range(N)], kind="stable")
    g = None
    for s in range(step):
        ids = order[BATCH * s:BATCH * (s + 1)]
        g, _ = b.gradient(x[ids], t[ids])
        b.adam_step(g, LR)
    assert np.array_equal(a.get_params(), b.get_params())
    for net in (a, b):  # the next step's bias corrections are those of step + 1
        net.adam_step(np.linspace(-1.0, 1.0, p.CNN_PARAMS).astype(np.float32), LR)
    assert np.array_equal(a.get_params(), b.get_params())
    # and training goes on
    assert np.isfinite(a.train(1, BATCH, LR, SEED))
    a.close()
    b.close()
