"""A training step whose launches fail reports it and changes nothing: neither the weights
nor Adam's step count."""
import ctypes as C
import os
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")
dg = pytest.importorskip("paper_2404_08952_gb300")


@pytest.mark.gpu
def test_a_failed_gradient_leaves_weights_and_step():
    rng = np.random.default_rng(2)
    x = torch.from_numpy(rng.random((500, 24)).astype(np.float32)).cuda()
    y = torch.from_numpy((rng.random(500) < 0.3).astype(np.uint8)).cuda()
    nets = [dg.MLP(seed=3), dg.MLP(seed=3)]
    theta0 = nets[0].get_params()
    torch.cuda.synchronize()
    # a stream whose capture was invalidated (by waiting for it) takes no launches
    cu = C.CDLL("libcuda.so.1")
    s, g = C.c_void_p(), C.c_void_p()
    assert cu.cuStreamCreate(C.byref(s), 1) == 0
    assert cu.cuStreamBeginCapture_v2(s, 1) == 0
    assert cu.cuStreamSynchronize(s) != 0
    stream = torch.cuda.ExternalStream(s.value)
    with pytest.raises(dg.DolincError) as e:
        nets[0].train_step(x, y, 1e-3, 2.0, stream=stream)
    assert e.value.status == 4
    assert cu.cuStreamEndCapture(s, C.byref(g)) != 0 and not g.value
    assert cu.cuStreamDestroy_v2(s) == 0
    np.testing.assert_array_equal(nets[0].get_params(), theta0)
    for net in nets:
        net.train_step(x, y, 1e-3, 2.0)
    a, b = (net.get_params() for net in nets)
    assert np.abs(a - theta0).max() > 0
    np.testing.assert_array_equal(a, b)


def test_opt_in_to_large_shared_memory_is_made_per_device():
    """No process-wide flag decides whether the training and solver kernels are set up: the
    call that creates a handle on a device does it."""
    csrc = os.path.join(os.path.dirname(dg.__file__), "csrc")
    for name in ("indicator.cu", "implicit.cu"):
        assert not re.search(r"static bool attr", open(os.path.join(csrc, name)).read()), name
