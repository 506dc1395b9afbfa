"""The network's gradients with dense hidden layers: long sums of FP32 gradients in every
backward product, against plain PyTorch in FP64.

Inputs are 0 and +-1 and the hidden weights 0 and +-1, so that every activation is an
integer of at most 256: exact in BF16, and the reference rounds nowhere the path does not.
Tolerance in the 2-norm of each gradient: three FP32 stages follow one another (the output
gradient, 4e-7; the products, whose 24-bit operands and per-block FP32 sums add about 4e-7
each): 1.5e-6.  A product that kept one tensor-core accumulator over its whole K, which
is cut towards zero at every step, is off by 1.9e-6 (last layer, 512 rows) to 9e-6."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 1.5e-6


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


@pytest.mark.parametrize("batch,n_in,h1,h2,nv", [(512, 64, 256, 256, 4), (1024, 128, 192, 320, 2), (300, 50, 130, 200, 3)])
def test_dense_hidden_layers(pkg, batch, n_in, h1, h2, nv):
    g = torch.Generator(device="cuda").manual_seed(batch + h1)
    no = nv * n_in
    tri = lambda *s, p: (torch.rand(*s, device="cuda", generator=g) < p).float() * \
        torch.sign(torch.randn(*s, device="cuda", generator=g))
    W = [tri(n_in, h1, p=1.0), tri(h1, h2, p=0.5),
         (5e-4 * torch.randn(h2, no, device="cuda", generator=g)).bfloat16().float()]
    x = tri(batch, n_in, p=0.25)
    t = torch.randn(batch, nv, n_in, device="cuda", generator=g)
    t = (t / t.norm(dim=2, keepdim=True)).reshape(batch, no).contiguous()
    Wd, X = [w.double() for w in W], x.double()
    a1 = torch.relu(X @ Wd[0])
    a2 = torch.relu(a1 @ Wd[1])
    assert float(a1.max()) <= 256 and float(a2.max()) <= 256
    w = torch.softmax(8 * X, dim=1).sqrt()[:, None, :]
    y = (a2 @ Wd[2]).view(batch, nv, n_in) * w
    td = t.double().view(batch, nv, n_in)
    pt = (y * td).sum(-1)
    d3 = (2.0 / (batch * nv) * (y - torch.where(pt >= 0, 1.0, -1.0)[..., None] * td) * w).reshape(batch, -1)
    d2 = (d3 @ Wd[2].T) * (a2 > 0)
    d1 = (d2 @ Wd[1].T) * (a1 > 0)
    ref = [(X.T @ d1, d1.sum(0)), (a1.T @ d2, d2.sum(0)), (a2.T @ d3, d3.sum(0))]
    net = pkg.WarmStartNet(n_in=n_in, hidden=(h1, h2), n_vec=nv, batch_max=batch, seed=1)
    flat = net.get_params()
    flat.zero_()
    wo, bo = net.offsets()
    for l in range(3):
        flat[wo[l]:wo[l] + W[l].numel()] = W[l].reshape(-1)
    net.set_params(flat)
    _, grad = net.gradients(x, t)
    for l in range(3):
        for off, r in ((wo[l], ref[l][0]), (bo[l], ref[l][1])):
            got = grad[off:off + r.numel()].view(r.shape).double()
            assert float((got - r).norm()) <= TOL * float(r.norm()), (l, r.shape, float((got - r).norm() / r.norm()))
    net.close()
