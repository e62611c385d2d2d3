"""EnergyFn: the gradients are those of the system that forward saw, whatever
is written into the caller's list, elements and box before backward; and each
combination of wanted gradients gives the same ones."""
import numpy as np
import pytest
import torch

from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import EnergyFn, TensorNet
from tests.gpu_helpers import DEV

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]

N = 60


def _model():
    return TensorNet(synth.init_weights(synth.ModelShape(), seed=0), max_atoms=N, max_pairs=N * (N - 1), precision=2,
                     device=DEV)


def _systems():
    """Two placements of N atoms in boxes of their own, with their elements."""
    for seed, side in ((1, 12.0), (2, 12.5)):
        s = synth.random_cluster(N, seed=seed)
        yield (torch.from_numpy(s.pos).to(DEV), torch.from_numpy(np.ascontiguousarray(s.z)).to(DEV),
               torch.eye(3, device=DEV)[None] * side)


def _grads(m, w, pos, z, box):
    pos, w = pos.clone().requires_grad_(), w.clone().requires_grad_()
    E = EnergyFn.apply(pos, w, m, z, m.neighbors(pos.detach(), None, box), None, box, 1)
    return torch.autograd.grad(E.sum(), (pos, w))


@pytest.mark.parametrize("reuse", ["list", "all"])
def test_gradients_of_a_sum_over_one_reused_list(reuse):
    m = _model()
    w0 = m.weights.clone()
    systems = list(_systems())
    want = [_grads(m, w0, *s) for s in systems]
    w = w0.clone().requires_grad_()
    nl = m.neighbors(systems[0][0], None, systems[0][2])
    z, box = (t.clone() for t in systems[0][1:])
    leaves, total = [], 0.0
    for pos, zs, bs in systems:
        if reuse == "all":
            z.copy_(zs)
            box.copy_(bs)
        else:
            z, box = zs, bs
        leaves.append(pos.clone().requires_grad_())
        m.neighbors(pos, None, box, out=nl)
        total = total + EnergyFn.apply(leaves[-1], w, m, z, nl, None, box, 1).sum()
    nl.col.zero_()
    total.backward()
    for leaf, (gp, _) in zip(leaves, want):
        assert torch.equal(leaf.grad, gp)
    assert torch.equal(w.grad, want[0][1] + want[1][1])


def test_wanted_gradients_alone_and_together():
    m = _model()
    w0 = m.weights.clone()
    pos, z, box = next(_systems())
    gp, gw = _grads(m, w0, pos, z, box)
    nl = m.neighbors(pos, None, box)
    w = w0.clone().requires_grad_()
    EnergyFn.apply(pos, w, m, z, nl, None, box, 1).sum().backward()
    assert torch.equal(w.grad, gw)
    p = pos.clone().requires_grad_()
    (3 * EnergyFn.apply(p, w0, m, z, nl, None, box, 1).sum()).backward()
    # the pass that keeps weight gradients forms the same sums in another order
    scale = gp.square().mean().sqrt()
    assert ((p.grad / 3 - gp).square().mean().sqrt() <= 1e-5 * scale).item()
