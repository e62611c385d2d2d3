"""The failure path of the staged message kernels, made to happen without a
fault: with copying warps that bring nothing and every wait limited to 2,048
tries, the kernels record TIMEOUT (6), write nothing and return; the same call
without the hold then gives the sums of a plain FP64 evaluation."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2402_17660_gb300 import _lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")]


def _graph(n, rng):
    """A symmetric CSR (40% of all pairs) with the pair of each directed edge."""
    adj = np.triu(rng.random((n, n)) < 0.4, 1)
    i, j = np.nonzero(adj)
    pair = -np.ones((n, n), np.int32)
    pair[i, j] = pair[j, i] = np.arange(len(i))
    row_ptr = np.concatenate([[0], np.cumsum((pair >= 0).sum(1))])
    r, c = np.nonzero(pair >= 0)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.int32)).cuda()
    return dev(row_ptr), dev(c), dev(pair[r, c]), torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda()


@pytest.mark.parametrize("F", [64, 128])
@pytest.mark.parametrize("backward", [0, 1])
def test_waits_run_out_and_leave_the_context_usable(F, backward):
    n = 200
    row_ptr, col, pair_of, i, j = _graph(n, np.random.default_rng(1))
    U = len(i)
    g = torch.Generator(device="cuda").manual_seed(F)
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda")
    a3, phi, V, V2 = rand(U, 3, F), torch.rand(U, generator=g, device="cuda"), rand(9 * n, F), rand(9 * n, F)
    start = rand(9 * n, F)
    lib = _lib.load()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def call(limit, hold):
        out, ga3, gphi = start.clone(), torch.full((U, 3, F), float("nan"), device="cuda"), torch.zeros(2, U, device="cuda")
        status.zero_()
        rc = lib.tnet_debug_message_tile(F, backward, n, p(row_ptr), p(col), p(pair_of), p(a3), p(phi), p(V), p(V2),
                                         p(out), p(ga3), p(gphi), U, limit, hold, p(status),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        return rc, int(status.item()), out, ga3, gphi

    assert call(0, 1)[0] == 1   # a hold without a limit of its own is refused
    rc, code, out, ga3, gphi = call(2048, 1)
    assert rc == 0 and code == 6
    assert torch.equal(out, start) and ga3.isnan().all() and not gphi.any()
    rc, code, out, ga3, gphi = call(0, 0)
    assert rc == 0 and code == 0
    plane = torch.tensor([0] + [1] * 3 + [2] * 5, device="cuda")
    at = lambda X: torch.cat([X[:n].view(n, 1, F), X[n:4 * n].view(n, 3, F), X[4 * n:].view(n, 5, F)], 1).double()
    v, v2, a = at(V), at(V2), a3.double()
    f = (phi.double()[:, None, None] * torch.nn.functional.silu(a))[:, plane]
    want = at(start) if backward else torch.zeros(n, 9, F, dtype=torch.float64, device="cuda")
    want = want.index_add(0, i, f * v[j]).index_add(0, j, f * v[i])
    size = want.abs().new_zeros(n, 9, F).index_add(0, i, (f * v[j]).abs()).index_add(0, j, (f * v[i]).abs())
    # rows of about 80 terms, each rounded a few times and added in one chain
    tol = 200 * 2.0 ** -24
    assert ((at(out) - want).abs() <= tol * (size + want.abs())).all()
    if backward:
        prod = v[i] * v2[j] + v[j] * v2[i]
        mag = (v[i] * v2[j]).abs() + (v[j] * v2[i]).abs()
        per = lambda x: torch.stack([x[:, plane == k].sum(1) for k in range(3)], 1)
        s = torch.sigmoid(a)
        ds = phi.double()[:, None, None] * s * (1 + a * (1 - s))
        assert ((ga3.double() - per(prod) * ds).abs() <= tol * per(mag) * (ds.abs() + phi.double()[:, None, None])).all()
        gp = (per(prod) * a * s).sum((1, 2))
        assert ((gphi.double().sum(0) - gp).abs() <= tol * (per(mag) * (a * s).abs()).sum((1, 2))).all()
