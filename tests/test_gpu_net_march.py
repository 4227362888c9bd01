"""The marching tensor-core kernels of the network (k_net.cu): waits that run
out part of the way, at poll bounds between none and enough."""
import pytest
import torch

from paper_1602_08847_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def netmod(lib):
    from paper_1602_08847_gb300 import net
    return net


@pytest.mark.parametrize("polls", [1, 2, 3, 5, 8, 13, 30, 100, 1000])
def test_waits_that_run_out_midway(netmod, polls):
    """With a small poll bound some warps give up and others do not, at any of
    the waits.  Every call returns, either with the result of an undisturbed
    run or with a give-up on record, and the next undisturbed run is right."""
    shape, K = (9, 70, 90), 2                 # 540 tiles: several a block, runs that cross columns
    theta = torch.from_numpy(synth.net_init(31, K).astype("float32")).cuda()
    y = torch.from_numpy(synth.random_field(shape, 32, -0.3, 1.0).astype("float32")).cuda()
    ta = torch.zeros((shape[0], K - 1, shape[1], shape[2]), dtype=torch.bfloat16, device="cuda")
    a = torch.relu(torch.from_numpy(synth.random_field(shape + (32,), 33).astype("float32"))).cuda().bfloat16()
    w = torch.from_numpy(synth.random_field((32, 32, 3, 3, 3), 34, -0.1, 0.1).astype("float32")).cuda()
    n = netmod.WarmStartNet(shape, training=True, theta=theta, n_out=K)

    def calls():
        yield lambda: (netmod.conv3d_forward(a, w, None, True),)
        yield lambda: (netmod.conv3d_backward_data(a, w, None),)
        yield lambda: netmod.conv3d_backward_weights(a, a)
        yield lambda: (n.loss_grad(y, torch.relu(y), ta)[1],)

    def guarded(f):
        try:
            out = f()
        except netmod._m.MuffinError as e:
            assert "TIMEOUT" in str(e)        # loss_grad reports (and clears) the give-ups itself
            return None
        torch.cuda.synchronize()
        return None if netmod.wait_timeouts() else out

    refs = [f() for f in calls()]
    assert netmod.wait_timeouts() == 0
    for f, ref in zip(calls(), refs):
        try:
            netmod.set_wait_limit(polls)
            got = guarded(f)
        finally:
            netmod.set_wait_limit(None)
        assert got is None or all(torch.equal(p, q) for p, q in zip(got, ref))
        assert all(torch.equal(p, q) for p, q in zip(f(), ref))
        assert netmod.wait_timeouts() == 0
    n.close()
