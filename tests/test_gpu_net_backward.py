"""The warm-start network's backward products (three BF16 parts of the FP32 gradient on the
tensor cores) at the edges of their tiles: widths that are no multiple of 64 or of 8, one row,
64 and 65 rows, an output narrower than a tile, more rows than one backward chunk (4096),
unaligned user arrays.

The hidden layers are permutations with signs and the inputs BF16 values, so that every
activation is exact in BF16 and the reference below (plain PyTorch, FP64) rounds nowhere the
path does not.  Tolerance: the output gradient is formed in FP32 from a sum of up to 256
products (about sqrt(256) 2^-24 = 1e-6 relative) and two more such sums follow: 5e-6 in the
2-norm of each gradient."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 5e-6


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


def make(pkg, batch, n_in, h1, h2, nv, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    net = pkg.WarmStartNet(n_in=n_in, hidden=(h1, h2), n_vec=nv, batch_max=batch, seed=1)
    no = nv * n_in
    W = [torch.zeros(n_in, h1, device="cuda"), torch.zeros(h1, h2, device="cuda"), (0.05 * rnd(h2, no)).bfloat16().float()]
    W[0][torch.arange(h1, device="cuda") % n_in, torch.arange(h1, device="cuda")] = torch.sign(rnd(h1))
    W[1][torch.randint(0, h1, (h2,), device="cuda", generator=g), torch.arange(h2, device="cuda")] = 1.0
    flat = net.get_params()
    flat.zero_()
    wo, bo = net.offsets()
    for l in range(3):
        flat[wo[l]:wo[l] + W[l].numel()] = W[l].reshape(-1)
    net.set_params(flat)
    x = (0.5 * rnd(batch, n_in)).bfloat16().float()
    t = rnd(batch, nv, n_in)
    t = (t / t.norm(dim=2, keepdim=True)).reshape(batch, no).contiguous()
    return net, W, x, t


def reference(W, x, t, nv):
    B, n_in = x.shape
    Wd, X = [w.double() for w in W], x.double()
    h1 = torch.relu(X @ Wd[0])
    h2 = torch.relu(h1 @ Wd[1])
    w = torch.softmax(8 * X, dim=1).sqrt()[:, None, :]
    y = (h2 @ Wd[2]).view(B, nv, n_in) * w
    td = t.double().view(B, nv, n_in)
    pt = (y * td).sum(-1)
    loss = ((y * y).sum(-1) + (td * td).sum(-1) - 2 * pt.abs()).mean()
    d = (2.0 / (B * nv) * (y - torch.where(pt >= 0, 1.0, -1.0)[..., None] * td) * w).reshape(B, -1)
    d2 = (d @ Wd[2].T) * (h2 > 0)
    d1 = (d2 @ Wd[1].T) * (h1 > 0)
    return y.reshape(B, -1), loss, [X.T @ d1, h1.T @ d2, h2.T @ d], [d1.sum(0), d2.sum(0), d.sum(0)]


@pytest.mark.parametrize("batch,n_in,h1,h2,nv", [
    (1, 64, 64, 64, 1), (64, 64, 128, 192, 3), (65, 128, 64, 256, 2), (300, 64, 320, 64, 5),      # tensor-core forward
    (17, 27, 50, 33, 1), (63, 216, 130, 129, 3), (129, 30, 72, 200, 2),                            # CUDA-core forward
    (4100, 64, 64, 128, 2)])                                                                       # two chunks
def test_gradients_against_fp64(pkg, batch, n_in, h1, h2, nv):
    net, W, x, t = make(pkg, batch, n_in, h1, h2, nv)
    y_ref, loss_ref, gw, gb = reference(W, x, t, nv)
    y = net.forward(x)
    assert float((y.double() - y_ref).norm() / y_ref.norm()) < TOL
    loss, grad = net.gradients(x, t)
    assert loss == pytest.approx(float(loss_ref), rel=TOL)
    wo, bo = net.offsets()
    for l in range(3):
        for off, ref in ((wo[l], gw[l]), (bo[l], gb[l])):
            got = grad[off:off + ref.numel()].view(ref.shape).double()
            assert float((got - ref).norm()) <= TOL * float(ref.norm()) + 1e-30, (l, ref.shape)
    net.close()


@pytest.mark.parametrize("n_in,h1,h2,nv", [(64, 64, 128, 2), (27, 40, 33, 2)])
def test_unaligned_arrays_and_row_counts_in_turn(pkg, n_in, h1, h2, nv):
    """Outputs at 4-byte aligned addresses, and calls whose row count changes, give the bits
    of the aligned call."""
    net, W, x, t = make(pkg, 130, n_in, h1, h2, nv)
    y, (loss, grad) = net.forward(x), net.gradients(x, t)
    yu = torch.empty(y.numel() + 1, device="cuda")[1:].view(y.shape)
    gu = torch.zeros(grad.numel() + 1, device="cuda")[1:]
    pkg.msmg_net_forward(net.handle, x, yu)
    pkg.msmg_net_gradients(net.handle, x[:70].contiguous(), t[:70].contiguous())
    net.forward(x[:5].contiguous())
    lu = pkg.msmg_net_gradients(net.handle, x, t, gu)
    assert torch.equal(y, yu) and loss == lu
    wo, bo = net.offsets()
    for l, (a, b) in enumerate(((n_in, h1), (h1, h2), (h2, nv * n_in))):
        assert torch.equal(grad[wo[l]:wo[l] + a * b], gu[wo[l]:wo[l] + a * b])
        assert torch.equal(grad[bo[l]:bo[l] + b], gu[bo[l]:bo[l] + b])
    net.close()


def test_parts_hold_extreme_gradients(pkg):
    """Targets scaled by 1e18 and 1e-18: the gradients keep their relative accuracy."""
    net, W, x, t = make(pkg, 64, 64, 64, 64, 2)
    for s in (1e18, 1e-18):
        ts = t * s
        _, _, gw, _ = reference(W, x, ts, 2)
        _, grad = net.gradients(x, ts)
        wo, _ = net.offsets()
        got = grad[wo[2]:wo[2] + gw[2].numel()].view(gw[2].shape).double()
        assert float((got - gw[2]).norm() / gw[2].norm()) < TOL
    net.close()
