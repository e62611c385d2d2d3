"""Bias gradients of a wide model over many rows: 20,000 atoms of one element,
none within the cutoff of another, have the same gradients, so each bias
gradient is 20,000 times that of one atom.  A column is summed in 32-row
blocks, the blocks of a row range in order and the ranges in order; with six
ranges or more (outputs of 48 tiles on 152 SMs) no more than 31 + 104 + 5
roundings meet one sum."""
import itertools

import numpy as np
import pytest
import torch

from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import NeighborList, TensorNet, unpack_weights

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]


def test_bias_gradients_of_many_equal_rows():
    F, K, n = 512, 8, 20_000
    W = synth.init_weights(synth.ModelShape(F=F, K=K, L=0), seed=0)
    dev = torch.device("cuda:0")
    m = TensorNet(W, F=F, K=K, L=0, max_atoms=n, max_systems=2, max_pairs=64, device=dev)
    pos = torch.tensor(list(itertools.islice(itertools.product(range(28), repeat=3), n)), device=dev).float() * 6.0
    z = torch.full((n,), 6, dtype=torch.int32, device=dev)
    batch = (torch.arange(n, device=dev) > 0).int()   # the first atom is a system of its own
    nl = NeighborList(torch.zeros(n + 1, dtype=torch.int32, device=dev), torch.zeros(64, dtype=torch.int32, device=dev),
                      torch.zeros(1, dtype=torch.int64, device=dev), 5.0)
    got = {}
    for name, seed in (("one", [1.0, 0.0]), ("all", [1.0, 1.0])):
        _, _, G = m.energy_forces(z, pos, nl, batch, None, 2, forces=False, grad_weights=True,
                                  seed=torch.tensor(seed, device=dev))
        m.check_status(name)
        got[name] = unpack_weights(G.cpu().numpy(), F, K, 0, 100)
    checked = 0
    for name in ("out_b", "head1_b", "head2_b"):
        one = got["one"][name].astype(np.float64)
        err = np.abs(got["all"][name] - n * one)
        assert (err <= (31 + 104 + 5 + 1) * 2.0 ** -24 * n * np.abs(one)).all(), (name, (err / (n * np.abs(one))).max())
        checked += np.count_nonzero(one)
    assert checked >= F
