"""The deepest model a descriptor allows (eight layers): one launch prepares
142 weight copies in BF16 mode.  Against the FP64 oracle at the repository's
BF16 tolerance, and the FP32 mode at its own."""
import pytest
import torch

from oracle.tensornet import TensorNet as Oracle
from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import TensorNet
from tests.gpu_helpers import (BF16_E_TOL, BF16_F_TOL, DEV, E_TOL, F_TOL, energy_errors, force_errors, gpu_pairs,
                               to_dev)

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]


@pytest.mark.parametrize("precision,e_tol,f_tol", [(0, E_TOL, F_TOL), (1, BF16_E_TOL, BF16_F_TOL)])
def test_eight_layers(precision, e_tol, f_tol):
    shape = synth.ModelShape(F=64, L=8)
    W = synth.init_weights(shape, seed=3)
    s = synth.random_cluster(40, seed=3)
    m = TensorNet(W, F=64, L=8, max_atoms=40, max_pairs=1600, precision=precision, device=DEV)
    nl = gpu_pairs(m, s)
    z, pos, _, _ = to_dev(s)
    E, Fg = m.energy_forces(z, pos, nl)[:2]
    m.check_status("energy_forces")
    Es, Ei, Fo = Oracle(W, F=64, L=8, rc=shape.cutoff_upper).energy_forces(s.z, s.pos, s.batch, s.box,
                                                                          n_systems=1)[:3]
    assert energy_errors(E.cpu().numpy(), Es, Ei, s.batch).max() <= e_tol
    assert force_errors(Fg.cpu().numpy(), Fo)[0] <= f_tol
