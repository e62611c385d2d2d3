"""The workspace that tnet_workspace_bytes asks for holds the weight operands
of the tensor-core modes: for every model shape, against a list of the
operands written down here.  On a GPU, deep 3xTF32 models against the oracle."""
import ctypes
import itertools

import pytest
import torch

from paper_2402_17660_gb300 import _lib, synth
from paper_2402_17660_gb300.tnet import TensorNet


def _up(n):
    return (n + 255) // 256 * 256


def _operand_bytes(F, K, L, precision, table):
    H = F // 2
    node = [3 * F * F] * (1 + 2 * L)                                     # mixing weights
    pair = [] if table else [2 * F * F, 6 * F * F] * L                   # radial layers 2 and 3
    basis = [] if table else [F * K] * L + [3 * F * K]                   # K-deep: always 3xTF32
    atom = [2 * F * F, 6 * F * F, 3 * F * F, H * F] if precision == 1 else []
    split = sum(4 * _up(4 * n) for n in basis + atom)                    # high and low part, forward and transposed
    if precision == 2:
        return split + sum(4 * _up(4 * n) for n in node + pair)
    return split + sum(2 * _up(2 * n) for n in node + pair)


def _bytes(lib, F, K, L, max_z, precision, table):
    d = _lib.ModelDesc(F, K, L, max_z, 5.0, 0.0, precision, 0, table)
    return lib.tnet_workspace_bytes(ctypes.byref(d), 1, 1, 0)


def test_weight_operands_fit_for_every_model_shape():
    lib = _lib.load()
    short = []
    for F, K, L, max_z, precision, table in itertools.product(
            range(64, 513, 64), (8, 16, 32, 64), range(9), (1, 100, 128), (1, 2), (0, 256)):
        have = _bytes(lib, F, K, L, max_z, precision, table) - _bytes(lib, F, K, L, max_z, 0, table)
        if precision == 1:   # less the bf16 copies of activations (one atom, one pair)
            layers = max(L, 1)
            have -= _up(18 * F)
            have -= 0 if table else _up(2 * F * layers) + _up(4 * F * layers) + _up(6 * F) + _up(4 * F)
        if have < _operand_bytes(F, K, L, precision, table):
            short.append((F, K, L, max_z, precision, table))
    assert not short, (len(short), short[:5])


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")
@pytest.mark.parametrize("F,L", [(64, 8), (128, 3), (128, 8), (256, 3)])
def test_deep_models_in_3xtf32(F, L):
    from oracle.tensornet import TensorNet as Oracle
    from tests.gpu_helpers import DEV, E_TOL, F_TOL, energy_errors, force_errors, gpu_pairs, to_dev
    shape = synth.ModelShape(F=F, L=L)
    W = synth.init_weights(shape, seed=3)
    s = synth.random_cluster(40, seed=3)
    m = TensorNet(W, F=F, L=L, max_atoms=40, max_pairs=1600, precision=2, device=DEV)
    nl = gpu_pairs(m, s)
    z, pos, _, _ = to_dev(s)
    E, Fg = m.energy_forces(z, pos, nl)[:2]
    m.check_status("energy_forces")
    Es, Ei, Fo = Oracle(W, F=F, L=L, rc=shape.cutoff_upper).energy_forces(s.z, s.pos, s.batch, s.box, n_systems=1)[:3]
    assert energy_errors(E.cpu().numpy(), Es, Ei, s.batch).max() <= E_TOL
    assert force_errors(Fg.cpu().numpy(), Fo)[0] <= F_TOL
