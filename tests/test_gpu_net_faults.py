"""GPU: waits inside the network's convolution kernels that run out of time
(S3TTV_NET_OPT_WAIT_NS) end the call with S3TTV_ECUDA and leave the context and
the network usable.  Under a limit of zero no wait is sat out and the call
ends so in any case; under a short one some waits run out, with products and copies
in flight, or none does."""
import numpy as np
import pytest

from test_gpu_unet import P, bf16_params  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one and two tiles along H, weights resident (32 channels) and streamed (64 and more)
SHAPES = [(1, 4, 4, 4), (3, 24, 36, 28)]


def volumes(shape):
    g = torch.Generator().manual_seed(5)
    return [torch.rand(shape, generator=g).cuda() for _ in range(4)]


def equal(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("shape", SHAPES)
def test_waits_that_run_out_are_reported_and_leave_the_network_usable(P, shape):  # noqa: F811
    args = volumes(shape)
    with P.WarmStartNet(0) as net:
        net.set_params(bf16_params(21))
        before = net.forward(args[0])
        loss = net.gradient(*args)[0]
        net.set_option(P.NET_OPT_WAIT_NS, 0)
        for call in (lambda: net.forward(args[0]), lambda: net.gradient(*args)):
            with pytest.raises(P.S3TTVError) as e:
                call()
            assert e.value.status == P.ECUDA and "time" in str(e.value)
        for ns in (1, 500, 2000, 10000, 50000):
            net.set_option(P.NET_OPT_WAIT_NS, ns)
            for call in (lambda: net.forward(args[0]), lambda: net.gradient(*args)):
                try:
                    out = call()
                except P.S3TTVError as err:
                    assert err.status == P.ECUDA
                else:
                    assert equal(out, before) if len(out) == 3 else out[0] == pytest.approx(loss, rel=1e-12)
        net.set_option(P.NET_OPT_WAIT_NS, 4e9)
        assert equal(net.forward(args[0]), before)
        assert net.gradient(*args)[0] == pytest.approx(loss, rel=1e-12)
        assert np.isfinite(net.gradient(*args)[1]).all()


def test_time_limit_is_checked(P):  # noqa: F811
    with P.WarmStartNet(0) as net:
        for key, value in ((P.NET_OPT_WAIT_NS, -1.0), (P.NET_OPT_WAIT_NS, float("nan")), (P.NET_OPT_WAIT_NS, 1e12),
                           (99, 1.0)):
            with pytest.raises(P.S3TTVError) as e:
                net.set_option(key, value)
            assert e.value.status == P.EINVAL


def test_no_training_step_along_a_failed_gradient(P):  # noqa: F811
    """A step whose gradient fails leaves parameters, moments and step count alone: the
    steps around it give what they give without it (they differ in the order of the
    gradient's FP32 additions: 1e-3 of a step, as Adam divides a gradient by its size;
    a step along the cut-off gradient moves parameters by 1e-3 = lr each)."""
    args = volumes((2, 8, 8, 8))
    runs = []
    for fail in (False, True):
        with P.WarmStartNet(0) as net:
            net.set_params(bf16_params(23))
            net.train_step(*args, 1e-3)
            if fail:
                before = net.get_params()
                net.set_option(P.NET_OPT_WAIT_NS, 0)
                with pytest.raises(P.S3TTVError) as e:
                    net.train_step(*args, 1e-3)
                assert e.value.status == P.ECUDA
                net.set_option(P.NET_OPT_WAIT_NS, 4e9)
                np.testing.assert_array_equal(net.get_params(), before)
            loss = net.train_step(*args, 1e-3)
            runs.append((loss, net.get_params()))
    assert runs[0][0] == pytest.approx(runs[1][0], rel=1e-4)
    moved = np.abs(runs[0][1] - runs[1][1])
    assert np.mean(moved <= 1e-6) >= 0.99
