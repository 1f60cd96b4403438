"""The run-merged scatter (scatter_runs) against the FP64 oracle where its walk takes each of its
branches: particles in the caller's order (mpm_step_noalloc does not sort) ascending and
descending along the last axis, in steps of two nodes, all in one cell, and in random order, at
counts around the edges of a walk, a warp and a tile."""
import numpy as np
import pytest

import oracle
from mpm_testlib import rel_l2, to_np
from paper_1910_00935_gb300 import scenes
from test_gpu_parity import POS_TOL, _compare_grads, _compare_states, _oracle_grad_linear, _oracle_states, _random_seeds

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


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("kind", ["off the grid", "inverted"])
def test_refused_particle_adds_nothing(mpm, dim, kind):
    """A particle whose stencil leaves the grid, or whose det F <= 0, is skipped wherever it stands in a
    warp: the others come out as in a run without it (one-step bars)."""
    n, n_grid = 70, 64
    x = _positions(dim, "ascending", n, 1.0 / n_grid).astype(np.float32)
    u = lambda s, rows: (scenes.uniform(6, s, rows * n).reshape(rows, n) * 2 - 1).astype(np.float32)  # noqa: E731
    F = (np.eye(dim).reshape(-1, 1) + 0.02 * u(3, dim * dim)).astype(np.float32)
    good = np.concatenate([x, u(1, dim), 3.0 * u(2, dim * dim), F])

    def step(st):
        N = st.shape[1]
        desc = dict(dim=dim, n_grid=n_grid, n_particles=[N], dt=1e-4, material=mpm.MPM_NEO_HOOKEAN)
        st = torch.as_tensor(np.ascontiguousarray(st)).cuda()
        out, err = torch.full_like(st, float("nan")), torch.zeros(1, dtype=torch.int32, device="cuda")
        E, nu = torch.full((N,), 2e3, device="cuda"), torch.full((N,), 0.3, device="cuda")
        assert mpm.mpm_step_noalloc(mpm.make_desc(desc), st, E, nu, out, err) == mpm.MPM_OK
        return to_np(out), int(err.item())

    for bad in range(34):
        st = good.copy()
        if kind == "inverted":
            st[2 * dim + dim * dim, bad] *= -1.0
        else:
            st[0, bad] = 0.2 / n_grid  # stencil base -1
        got, err = step(st)
        assert err == (2 if kind == "inverted" else 1)
        want, none = step(np.delete(good, bad, 1))
        assert none == 0
        got = np.delete(got, bad, 1)
        for name, rows in (("x", slice(0, dim)), ("v", slice(dim, 2 * dim)), ("C", slice(2 * dim, 2 * dim + dim * dim)),
                           ("F", slice(2 * dim + dim * dim, None))):
            assert rel_l2(got[rows], want[rows]) <= TOL[name], (bad, name, rel_l2(got[rows], want[rows]))


@pytest.mark.parametrize("name,kw", [("cube3d", dict(n_side=11, n_grid=48)), ("square2d", dict(n_side=33))])
def test_refused_particle_adds_nothing_to_states_and_gradients(mpm, name, kw):
    """The same over a run and its reverse: the particle sorts first, at the head of the first warp's
    walk; deterministic sums, so the others' states and gradients are bitwise those without it."""
    T = 6

    def run(with_bad):
        scene = scenes.make(name, **kw)
        d, a = scene["desc"], scene["arrays"]
        d["deterministic_p2g"], d["ckpt_every"] = 1, 4
        seeds = _random_seeds(scene, np.random.default_rng(4))
        if with_bad:
            for k in ("x0", "v0", "C0", "F0", "E", "nu"):
                a[k] = np.ascontiguousarray(np.concatenate([a[k][..., :1], a[k]], -1))
            a["x0"][:, 0] = 0.2 / d["n_grid"]
            d["n_particles"] = [d["n_particles"][0] + 1]
            seeds = {k: np.concatenate([np.zeros_like(v[:, :1]), v], 1) for k, v in seeds.items()}
        sim = mpm.from_scene(scene, max_steps=T)
        sim.forward(T)
        out = [t.clone() for t in sim.state()]
        out += [v for k, v in sim.backward(**{k: torch.as_tensor(v) for k, v in seeds.items()}).items() if k != "gw"]
        rc = mpm.mpm_sync_status(sim.h)
        assert rc == (mpm.MPM_ERR_OOB if with_bad else mpm.MPM_OK)
        sim.close()
        return out

    for got, want in zip(run(True), run(False)):
        assert torch.equal(got[..., 1:], want)


@pytest.mark.parametrize("name,kw", [("cube3d", dict(n_side=14, n_grid=48)), ("rects2d", dict(n_scenes=3, n_min=300, n_max=1500)),
                                     ("robots3d", dict(n_scenes=2, dims=(12, 8, 8)))])
@pytest.mark.parametrize("order", [0, 1, 2])
@pytest.mark.parametrize("gather,det", [(512, 0), (0, 0), (512, 1), (0, 1)])
def test_particle_orders_match_oracle(mpm, name, kw, order, gather, det):
    """The walk's merging depends on the order of the particles, its sums do not."""
    scene, T = scenes.make(name, **kw), 6
    scene["desc"]["ckpt_every"], scene["desc"]["deterministic_p2g"] = 3, det
    seeds = _random_seeds(scene, np.random.default_rng(21))
    sim = mpm.from_scene(scene, max_steps=T)
    sim.set_option(mpm.MPM_OPT_GATHER_CAPACITY, gather)
    sim.set_option(mpm.MPM_OPT_SORT_ORDER, order)
    sim.reload()
    sim.forward(T)
    state = [to_np(t) for t in sim.state()]
    grad = {k: to_np(v) for k, v in sim.backward(**{k: torch.as_tensor(v) for k, v in seeds.items()}).items()}
    assert mpm.mpm_sync_status(sim.h) == mpm.MPM_OK
    sim.close()
    _compare_states(state, _oracle_states(scene, T), scene, POS_TOL)
    keys = ["gx0", "gv0", "gC0", "gF0", "gE", "gnu"] + (["gw"] if scene["desc"]["n_groups"] else [])
    _compare_grads(grad, _oracle_grad_linear(scene, T, {k: v.astype(np.float64) for k, v in seeds.items()}), keys)
