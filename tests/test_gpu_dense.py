"""The FP32 GEMM's four tile sizes and the weight-gradient tiles at the shapes
where they can go wrong: channel counts that do not fill a 128-wide tile, a
basis size that is no multiple of 32, row counts below and just past a tile,
and enough pairs for the 128 x 128 tile.  Energies, forces and every weight
gradient are held to the FP64 oracle at the repository's tolerances."""
import numpy as np
import pytest
import torch

from oracle.tensornet import TensorNet as Oracle
from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import TensorNet, unpack_weights
from tests.gpu_helpers import DEV, E_TOL, F_TOL, energy_errors, force_errors, gpu_pairs, to_dev

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]


# atoms of a cluster at the density of the 32-atom molecule: 3 (one pair's
# worth of rows), 33 and 129 (just past 32 and 128 rows), 700 (about 13,000
# pairs: 128-wide tiles at F = 192, two per SM from 320 columns on)
@pytest.mark.parametrize("n,F,K", [(3, 64, 8), (33, 64, 24), (33, 192, 40), (129, 192, 16), (700, 192, 24)])
def test_dense_layers_against_oracle(n, F, K):
    shape = synth.ModelShape(F=F, K=K, L=1)
    W = synth.init_weights(shape, seed=1)
    s = synth.random_cluster(n, seed=n)
    m = TensorNet(W, F=F, K=K, L=1, max_atoms=n, max_pairs=max(64, min(n * n, 80 * n)), device=DEV)
    nl = gpu_pairs(m, s)
    z, pos, _, _ = to_dev(s)
    E, Fg, G = m.energy_forces(z, pos, nl, grad_weights=True)
    m.check_status("energy_forces")
    o = Oracle(W, F=F, K=K, L=1, rc=shape.cutoff_upper)
    Es, Ei, Fo, Go = o.energy_forces(s.z, s.pos, s.batch, s.box, n_systems=1, want_weights=True)
    assert energy_errors(E.cpu().numpy(), Es, Ei, s.batch).max() <= E_TOL
    assert force_errors(Fg.cpu().numpy(), Fo)[0] <= F_TOL
    for name, g in unpack_weights(G.cpu().numpy(), F, K, 1, shape.max_z).items():
        ref = np.asarray(Go[name], np.float64)
        scale = np.sqrt(np.mean(ref ** 2))
        err = np.sqrt(np.mean((g.astype(np.float64) - ref) ** 2))
        assert err <= F_TOL * scale if scale > 0 else err == 0, (name, err, scale)
