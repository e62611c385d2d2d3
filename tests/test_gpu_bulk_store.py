"""The tensor-core GEMMs whose epilogue writes whole 32-row groups with bulk
tensor stores (radial layers, projections, channel mixing) at the edges of a
group: fewer rows than one, one row past a group or a tile, classes that start
inside a group, and channel counts of half a column tile or one and a half.
Against the FP64 oracle at the repository's tolerances for the FP32-accurate
mode."""
import pytest
import torch

from oracle.tensornet import TensorNet as Oracle
from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import TensorNet
from tests.gpu_helpers import DEV, E_TOL, F_TOL, energy_errors, force_errors, gpu_pairs, to_dev

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]


@pytest.mark.parametrize("F", [64, 128, 192])
@pytest.mark.parametrize("n", [3, 32, 33, 129])
def test_rows_at_group_edges(n, F):
    shape = synth.ModelShape(F=F, L=1)
    W = synth.init_weights(shape, seed=2)
    s = synth.random_cluster(n, seed=n)
    m = TensorNet(W, F=F, L=1, max_atoms=n + 5, max_pairs=max(64, min(n * n, 80 * n)) + 7, precision=2, device=DEV)
    nl = gpu_pairs(m, s)
    z, pos, _, _ = to_dev(s)
    E, Fg = m.energy_forces(z, pos, nl)[:2]
    m.check_status("energy_forces")
    Es, Ei, Fo = Oracle(W, F=F, L=1, rc=shape.cutoff_upper).energy_forces(s.z, s.pos, s.batch, s.box,
                                                                         n_systems=1)[:3]
    assert energy_errors(E.cpu().numpy(), Es, Ei, s.batch).max() <= E_TOL
    assert force_errors(Fg.cpu().numpy(), Fo)[0] <= F_TOL
