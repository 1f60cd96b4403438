"""The grids that a forward leaves for its backward (kept segment grids): whatever is called between
the two, or instead of one of them, gives what a fresh handle gives -- bitwise, in the
deterministic mode, where the order of the sums does not matter."""
import numpy as np
import pytest

from paper_1910_00935_gb300 import scenes
from test_gpu_parity import _random_seeds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

T = 14


@pytest.fixture(scope="module")
def mpm():
    from paper_1910_00935_gb300 import build, mpm as m
    build.build()
    return m


def _scene(name):
    s = {"cube": lambda: scenes.make("cube3d", n_side=12, n_grid=48),
         "rects": lambda: scenes.make("rects2d", n_scenes=3, n_min=200, n_max=700),
         "nn": lambda: scenes.make("robots_nn", n_scenes=2, dims=(12, 8, 8), hidden=8)}[name]()
    s["desc"]["deterministic_p2g"] = 1
    return s


def _back(sim, seeds):
    return [t.clone() for t in sim.backward(**seeds).values()]


def _same(a, b):
    assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("name", ["cube", "rects", "nn"])
@pytest.mark.parametrize("k", [4, 7, 40])  # a ragged last segment, an even one, one segment
@pytest.mark.parametrize("coarse", [0, 2])
def test_any_order_of_calls(mpm, name, k, coarse):
    scene = _scene(name)
    scene["desc"]["ckpt_every"], scene["desc"]["ckpt_coarse"] = k, coarse
    seeds = {key: torch.as_tensor(v).cuda() for key, v in _random_seeds(scene, np.random.default_rng(3)).items()}

    def fresh(steps, graphs=1):
        sim = mpm.from_scene(scene, max_steps=T)
        sim.set_option(mpm.MPM_OPT_USE_GRAPHS, graphs)
        sim.forward(steps)
        return sim

    ref_sim = fresh(T)
    ref = _back(ref_sim, seeds)
    sim9 = fresh(9, graphs=0)
    ref9 = _back(sim9, seeds)
    x = [t.clone() for t in ref_sim.state()]

    sim = fresh(T)
    sim.forward(T)                                  # a forward over the grids of another
    _same(_back(sim, seeds), ref)
    _same(_back(sim, seeds), ref)                   # a second backward of the same forward
    sim.forward(9)                                  # another length, other buffers
    sim.forward(T)
    sim.forward(9)
    _same(_back(sim, seeds), ref9)
    sim.forward(T)
    sim.reload()                                    # a set-up over kept grids
    sim.forward(T)
    _same(sim.state(), x)
    _same(_back(sim, seeds), ref)
    sim.forward(T)
    for option, value in ((mpm.MPM_OPT_GRID_RECOMPUTE, 1), (mpm.MPM_OPT_USE_GRAPHS, 0), (mpm.MPM_OPT_OVERLAP_RESIM, 0)):
        sim.set_option(option, value)               # an option between the two
        _same(_back(sim, seeds), ref)
        sim.forward(T)
        _same(_back(sim, seeds), ref)
    sim.set_option(mpm.MPM_OPT_GRID_RECOMPUTE, 0)
    sim.forward(T)
    _same(_back(sim, seeds), ref)
    assert mpm.mpm_sync_status(sim.h) == mpm.MPM_OK
    for s in (ref_sim, sim9, sim):
        s.close()


def test_diagnostic_grid_between(mpm):
    """mpm_initial_p2g_grid leaves a recorded forward, its kept grids among it, intact."""
    scene = scenes.make("cube3d", n_side=12, n_grid=48)
    scene["desc"]["ckpt_every"] = 40
    seeds = {key: torch.as_tensor(v).cuda() for key, v in _random_seeds(scene, np.random.default_rng(3)).items()}
    sim = mpm.from_scene(scene, max_steps=T)
    grid = torch.empty(1, 48 ** 3, 4, device="cuda")
    mpm.mpm_initial_p2g_grid(sim.h, grid)
    first = grid.clone()
    sim.forward(T)
    ref = _back(sim, seeds)
    sim.forward(T)
    mpm.mpm_initial_p2g_grid(sim.h, grid)
    assert float((grid - first).norm()) <= 1e-6 * float(first.norm())
    for a, b in zip(_back(sim, seeds), ref):
        assert float((a - b).norm()) <= 1e-4 * max(float(b.norm()), 1e-30)
    assert mpm.mpm_sync_status(sim.h) == mpm.MPM_OK
    sim.close()


@pytest.mark.parametrize("name", ["cube", "rects", "nn"])
@pytest.mark.parametrize("k", [4, 40])
@pytest.mark.parametrize("before", [False, True])  # a forward whose kept grids the capture meets
def test_calls_captured_by_the_caller(mpm, name, k, before):
    """A caller's own graph of a call, replayed any number of times and between calls made directly,
    gives what the call gives."""
    scene = _scene(name)
    scene["desc"]["ckpt_every"] = k
    seeds = {key: torch.as_tensor(v).cuda() for key, v in _random_seeds(scene, np.random.default_rng(3)).items()}
    ref_sim = mpm.from_scene(scene, max_steps=T)
    ref_sim.forward(T)
    x, ref = [t.clone() for t in ref_sim.state()], _back(ref_sim, seeds)

    sim = mpm.from_scene(scene, max_steps=T)
    sim.set_option(mpm.MPM_OPT_USE_GRAPHS, 0)  # (a library graph cannot be launched into a capture)
    out = [torch.empty_like(t) for t in x]
    g = {key: torch.empty_like(v) for key, v in ref_sim.backward(**seeds).items()}
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim.forward(T)
        _back(sim, seeds)
        if before:
            sim.forward(T)
    stream.synchronize()

    def capture(fn):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            fn()
        return graph

    def backward():
        mpm.mpm_backward(sim.h, **seeds, **{key: (v if v.numel() else None) for key, v in g.items()})

    forward = capture(lambda: (mpm.mpm_forward(sim.h, T), mpm.mpm_get_state(sim.h, *out)))
    both = capture(lambda: (mpm.mpm_forward(sim.h, T), backward()))
    setup = capture(lambda: mpm.mpm_set_initial(sim.h, *sim._inputs))
    sim.T = T

    def replay(graph):
        for t in out + list(g.values()):
            t.fill_(float("nan"))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()

    for _ in range(3):
        replay(forward)
        _same(out, x)
    for _ in range(2):
        replay(both)
        _same(list(g.values()), ref)
    replay(setup)
    replay(forward)
    _same(out, x)
    sim.reload()
    sim.forward(T)                      # called directly, a replay between it and its backward
    replay(forward)
    _same(_back(sim, seeds), ref)
    replay(forward)
    sim.forward(T)
    _same(_back(sim, seeds), ref)
    replay(both)
    _same(list(g.values()), ref)
    _same(_back(sim, seeds), ref)
    assert mpm.mpm_sync_status(sim.h) == mpm.MPM_OK
    ref_sim.close()
    sim.close()


@pytest.mark.parametrize("k", [4, 40])
@pytest.mark.parametrize("first,then", [(0, 1), (1, 0)])
def test_polar_cache_switched_between(mpm, k, first, then):
    """The factors that a forward leaves for its backward are used only where it wrote them."""
    scene = scenes.make("robots3d", n_scenes=2, dims=(12, 8, 8))
    scene["desc"]["deterministic_p2g"], scene["desc"]["ckpt_every"] = 1, k
    seeds = {key: torch.as_tensor(v).cuda() for key, v in _random_seeds(scene, np.random.default_rng(3)).items()}
    ref_sim = mpm.from_scene(scene, max_steps=T)
    ref_sim.forward(T)
    ref = _back(ref_sim, seeds)
    sim = mpm.from_scene(scene, max_steps=T)
    sim.set_option(mpm.MPM_OPT_POLAR_CACHE, first)
    sim.forward(T)
    sim.set_option(mpm.MPM_OPT_POLAR_CACHE, then)
    for _ in range(2):
        for a, b in zip(_back(sim, seeds), ref):  # (a factor formed in another pass may round differently)
            assert float((a - b).norm()) <= 1e-4 * float(b.norm())
    assert mpm.mpm_sync_status(sim.h) == mpm.MPM_OK
    ref_sim.close()
    sim.close()


def test_set_up_after_a_wait_that_gave_up_unseen(mpm):
    """A persistent forward whose barrier gives up leaves grids half written; a set-up clears them even if
    nobody asked for the status in between."""
    scene = scenes.make("square2d", n_side=32)
    scene["desc"]["deterministic_p2g"], scene["desc"]["ckpt_every"] = 1, 4  # (no grid of the early steps is kept)
    ref = mpm.from_scene(scene, max_steps=T)
    ref.forward(T)
    x = [t.clone() for t in ref.state()]
    sim = mpm.from_scene(scene, max_steps=T)
    sim.forward(T)  # (the grids are known to be clean from here on)
    first = list(sim._inputs)
    sim.set_initial(first[0] + 0.02, first[1] + 1.0, *first[2:6])
    sim.set_option(mpm.MPM_OPT_PERSISTENT, 1)
    sim.set_option(mpm.MPM_OPT_BARRIER_TIMEOUT_US, 20000)
    sim.set_option(mpm.MPM_OPT_BARRIER_TEST_EXTRA, 1)  # an arrival that never comes
    sim.forward(T)
    sim.set_option(mpm.MPM_OPT_PERSISTENT, 0)
    sim.set_initial(*first[:6])
    sim.forward(T)
    _same(sim.state(), x)
    assert mpm.mpm_sync_status(sim.h) == mpm.MPM_ERR_TIMEOUT  # (the wait that gave up is still reported)
    ref.close()
    sim.close()
