"""A training step whose products report a failure leaves the network as it was: masters,
Adam moments and step count.

The failure is the products' error word (a bounded wait that gave up sets it), set here by
the host before the call: the last 16 bytes the network takes of its workspace, which
msmg_net_workspace_size rounds up by 256.  Equal bits throughout: the same steps on the same
data."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


@pytest.mark.parametrize("n_in,hidden,nv", [(64, (64, 128), 2), (27, (50, 33), 3)])
@pytest.mark.parametrize("good", [0, 2])
def test_failed_step_is_not_applied(pkg, n_in, hidden, nv, good):
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(40, n_in, device="cuda", generator=g)
    t = torch.randn(40, nv * n_in, device="cuda", generator=g)
    kw = dict(n_in=n_in, hidden=hidden, n_vec=nv, batch_max=40, seed=2)
    plain, net = pkg.WarmStartNet(**kw), pkg.WarmStartNet(**kw)
    wo, bo = net.offsets()
    dims = (n_in,) + tuple(hidden) + (nv * n_in,)

    def params(m):
        p = m.get_params()
        return torch.cat([p[o:o + k] for l in range(3) for o, k in ((wo[l], dims[l] * dims[l + 1]), (bo[l], dims[l + 1]))])

    for _ in range(good):
        assert net.train_step(x, t, 1e-2) == plain.train_step(x, t, 1e-2)
    before, y = params(net), net.forward(x)
    net.workspace[-272:-268] = torch.tensor([1, 0, 0, 0], dtype=torch.uint8, device="cuda")
    with pytest.raises(pkg.MsmgError) as e:
        net.train_step(x, t, 1e-2)
    assert e.value.status == -11
    assert torch.equal(params(net), before) and torch.equal(net.forward(x), y)
    for _ in range(2):
        assert net.train_step(x, t, 1e-2) == plain.train_step(x, t, 1e-2)
        assert torch.equal(params(net), params(plain))
    net.close()
    plain.close()
