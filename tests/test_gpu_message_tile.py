"""The staged message kernels (one block per group of rows, node rows shared
through shared memory) at the sizes where their bookkeeping turns: fewer rows
than a group, group and grid remainders, rows without an edge, and rows longer
than one listing pass (which take several passes over the group).  Energies
equal those of the thread-per-channel form bit for bit (the same sums in the
same order); energies and forces are held to the FP64 oracle at the
repository's tolerances."""
import numpy as np
import pytest
import torch

from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import TensorNet
from tests.gpu_helpers import (DEV, E_TOL, F_TOL, energy_errors, force_errors, gpu_pairs, oracle_energy_forces,
                               to_dev)

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]

SHAPES = {F: synth.ModelShape(F=F) for F in (64, 128)}
WEIGHTS = {F: synth.init_weights(s, seed=0) for F, s in SHAPES.items()}
KNOB, STAGED, CHANNEL = 6, 3, 1


def _cloud(n, side, seed):
    """n atoms on a jittered lattice in a cube: dense enough for long rows"""
    rng = np.random.default_rng(seed)
    m = int(np.ceil(n ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    pos = (g + 0.5 + rng.uniform(-0.2, 0.2, (n, 3))) * (side / m)
    z = rng.choice(np.array([1, 6, 7, 8], np.int32), n)
    return synth.System(f"cloud{n}", z, pos.astype(np.float32), np.zeros(n, np.int32), None, 1)


# (atoms, cube side): group remainders of 6 and 12 rows; 130 and 280 atoms in
# 5 A have rows of up to 129 and about 270 active edges (two and three passes);
# 2,000 atoms pass one group per SM; 40 atoms in 60 A have none
@pytest.mark.parametrize("F", [64, 128])
@pytest.mark.parametrize("n,side", [(1, 3.0), (5, 4.0), (12, 5.0), (13, 5.0), (40, 60.0), (130, 5.0), (280, 5.0),
                                    (2000, 30.0)])
def test_staged_form(n, side, F):
    s = _cloud(n, side, seed=n)
    got = {}
    for form in (STAGED, CHANNEL):
        m = TensorNet(WEIGHTS[F], F=F, max_atoms=n, max_pairs=max(64, min(n * n, 600 * n)), device=DEV)
        knobs = m.get_tuning()
        knobs[KNOB] = form
        m.set_tuning(knobs)
        nl = gpu_pairs(m, s)
        z, pos, _, _ = to_dev(s)
        E, Fo, _ = m.energy_forces(z, pos, nl)
        m.check_status("energy_forces")
        got[form] = E.cpu().numpy(), Fo.cpu().numpy()
    assert np.array_equal(got[STAGED][0], got[CHANNEL][0])
    Es, Ei, Fo = oracle_energy_forces(WEIGHTS[F], s, SHAPES[F])
    E, Fg = got[STAGED]
    assert energy_errors(E, Es, Ei, s.batch).max() <= E_TOL
    if np.abs(Fo).max() > 0:
        assert force_errors(Fg, Fo)[0] <= F_TOL
    else:
        assert np.abs(Fg).max() == 0
