"""Pair lists that break the contract of tnet_energy_forces, in contexts whose
pair capacity is exactly the list's length: each is reported, only pairs with
both directed edges are evaluated, and the context stays good.  Half lists and
repeated columns hold more upper edges than the pair buffers (half the
capacity), and decreasing offsets make rows share edges."""
import numpy as np
import pytest
import torch

from oracle.neighbors import neighbor_pairs
from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import NeighborList, TensorNet
from tests.gpu_helpers import DEV, E_TOL, F_TOL, RC, force_error, to_dev

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]

W = synth.init_weights(synth.ModelShape(), seed=0)
N = 96


def _csr(i, j):
    """Rows in the given order of edges (i ascending)."""
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(i, minlength=N))])
    return row_ptr.astype(np.int32), np.asarray(j, np.int32)


def _lists(s):
    i, j = neighbor_pairs(s.pos, s.batch, s.box, RC)
    half = i < j
    yield "half", _csr(i[half], j[half]), None
    n = 5 * len(i) // 8   # what a search with that capacity hands on
    ti, tj = i[:n], j[:n]
    both = np.isin(tj * N + ti, ti * N + tj)
    yield "truncated", _csr(ti, tj), (ti[both], tj[both])
    row_ptr, col = _csr(i, j)
    yield "overlapping", (np.where(np.arange(N + 1) % 2 == 0, 0, len(col)).astype(np.int32), col), None
    a = np.argsort(np.linalg.norm(s.pos - s.pos[0], axis=1))[1:5]   # four neighbours of atom 0
    a = np.sort(a)
    m = 24
    yield "repeated", _csr(np.concatenate([np.zeros(4 * m, int), a]),
                           np.concatenate([np.tile(a, m), np.zeros(4, int)])), "any"
    yield "overlong", _csr(np.concatenate([np.zeros(N + 4, int), a]),
                           np.concatenate([np.tile(a, N // 4 + 1), np.zeros(4, int)])), None


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("name", ["half", "truncated", "overlapping", "repeated", "overlong"])
def test_malformed_list_is_reported_and_stays_inside_the_buffers(name, precision):
    s = synth.random_cluster(N, seed=12)
    (row_ptr, col), want = next((c, w) for k, c, w in _lists(s) if k == name)
    z, pos, _, _ = to_dev(s)

    def listed(rp, c):
        t = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.int32)).to(DEV)
        return NeighborList(t(rp), t(c), torch.tensor([len(c)], device=DEV), RC)

    m = TensorNet(W, max_atoms=N, max_pairs=len(col), precision=precision, device=DEV)

    def run(nl):
        m.reset_status()
        E, F, _ = m.energy_forces(z, pos, nl)
        torch.cuda.synchronize()
        return E.cpu().numpy(), F.cpu().numpy(), int(m.status.item())

    E, F, status = run(listed(row_ptr, col))
    assert status != 0
    assert np.isfinite(E).all() and np.isfinite(F).all()
    if want != "any":
        i, j = want if want is not None else (np.zeros(0, int), np.zeros(0, int))
        rp, c = _csr(i, j)
        E0, F0, status = run(listed(rp, np.append(c, np.zeros(1, int))))
        assert status == 0
        assert abs(E[0] - E0[0]) <= E_TOL * abs(E0[0])
        assert force_error(F, F0) <= F_TOL if np.any(F0) else not np.any(F)
    # the same context then evaluates a good list like one that never saw a bad one
    i, j = neighbor_pairs(s.pos[:16], s.batch[:16], None, RC)
    rp, c = _csr(i, j)
    assert len(c) <= len(col)
    E1, F1, status = run(listed(rp, c))
    clean = TensorNet(W, max_atoms=N, max_pairs=len(col), precision=precision, device=DEV)
    E2, F2, _ = clean.energy_forces(z, pos, listed(rp, c))
    assert status == 0
    assert np.array_equal(E1, E2.cpu().numpy()) and np.array_equal(F1, F2.cpu().numpy())
