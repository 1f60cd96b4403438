"""The run-merged scatter (scatter_runs) against the FP64 oracle where its walk takes each of its
branches: particles in the caller's order (mpm_step_noalloc does not sort) ascending and
descending along the last axis, in steps of two nodes, all in one cell, and in random order, at
counts around the edges of a walk, a warp and a tile."""
import numpy as np
import pytest

import oracle
from mpm_testlib import rel_l2, to_np
from paper_1910_00935_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one-step bars of the parity tests: x and F at 1e-5, v at 10x, C at 100x
TOL = {"x": 1e-5, "v": 1e-4, "C": 1e-3, "F": 1e-5}


@pytest.fixture(scope="module")
def mpm():
    from paper_1910_00935_gb300 import build, mpm as m
    build.build()
    return m


def _positions(dim, order, n, dx):
    r = scenes.uniform(5, dim, 2 * n * dim).reshape(2, dim, n)
    x = np.full((dim, n), 0.4) + 0.3 * dx * r[0]
    step = {"ascending": 0.5, "descending": -0.5, "by_two": 2.0, "one_cell": 0.0, "random": 0.0}[order]
    if order == "random":
        return 0.3 + 0.3 * r[1]
    k = np.arange(n)
    per_row = 24  # a row of 24, then the next row over
    x[-1] += (k % per_row) * step * dx - (0.2 if order == "by_two" else 0.0)  # 48 nodes stay inside
    x[0] += (k // per_row % 8) * 0.5 * dx
    return x


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("order", ["ascending", "descending", "by_two", "one_cell", "random"])
@pytest.mark.parametrize("n", [1, 3, 10, 11, 31, 32, 33, 127, 128, 129, 300])
def test_one_step_in_caller_order(mpm, dim, order, n):
    n_grid = 128 if dim == 2 else 64
    x = _positions(dim, order, n, 1.0 / n_grid).astype(np.float32)
    u = lambda s, rows: (scenes.uniform(6, s, rows * n).reshape(rows, n) * 2 - 1).astype(np.float32)  # noqa: E731
    v, C = u(1, dim), 3.0 * u(2, dim * dim)
    F = (np.eye(dim).reshape(-1, 1) + 0.02 * u(3, dim * dim)).astype(np.float32)
    E, nu = np.full(n, 2e3, np.float32), np.full(n, 0.3, np.float32)
    desc = dict(dim=dim, n_grid=n_grid, n_particles=[n], dt=1e-4, material=mpm.MPM_NEO_HOOKEAN)
    st = torch.as_tensor(np.concatenate([x, v, C, F])).cuda()
    out, err = torch.full_like(st, float("nan")), torch.zeros(1, dtype=torch.int32, device="cuda")
    assert mpm.mpm_step_noalloc(mpm.make_desc(desc), st, torch.as_tensor(E).cuda(), torch.as_tensor(nu).cuda(), out,
                                err) == mpm.MPM_OK
    assert int(err.item()) == 0
    out = to_np(out)
    f64 = [a.astype(np.float64) for a in (x, v, C, F)]
    mu, la = oracle.lame(E.astype(np.float64), nu.astype(np.float64))
    p = oracle.make_params(dim, n_grid, float(np.float32(1e-4)), (0.0, -9.8, 0.0), 3, oracle.NEO_HOOKEAN)
    ref = oracle.step(p, 0, *f64, mu, la)
    r0 = 0
    for name, want in zip("xvCF", ref):
        got = out[r0:r0 + want.shape[0]]
        r0 += want.shape[0]
        assert rel_l2(got, want) <= TOL[name], (name, rel_l2(got, want))
