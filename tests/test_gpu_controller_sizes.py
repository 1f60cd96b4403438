"""The closed-loop controller's kernels at the edges of their shapes -- one to eight groups, hidden
layers around the 32-lane and 64-unit limits, no time inputs, particles of every group and of none
mixed in each warp, an empty group, scenes of a few and of many tiles -- against the FP64 oracle, and
a scene alone against the same scene in a batch (bitwise, deterministic mode)."""
import numpy as np
import pytest

from paper_1910_00935_gb300 import scenes
from test_gpu_controller import KEYS
from test_gpu_parity import (POS_TOL, _compare_grads, _compare_states, _oracle_grad_linear, _oracle_states,
                             _random_seeds, _run_gpu)
from mpm_testlib import scene_slice, subset_scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mpm():
    from paper_1910_00935_gb300 import build, mpm as m
    build.build()
    return m


def _scene(dim, G, K, H, sides, seed=3):
    """Elastic squares or cubes whose particles belong to random groups (-1: none; the last group of
    several is left empty)."""
    parts = [scenes.make("square2d", n_side=n) if dim == 2 else scenes.make("cube3d", n_side=n, n_grid=64) for n in sides]
    s = parts[0]
    a, d = s["arrays"], s["desc"]
    for k in ("x0", "v0", "C0", "F0"):
        a[k] = np.ascontiguousarray(np.concatenate([p["arrays"][k] for p in parts], 1))
    for k in ("E", "nu"):
        a[k] = np.ascontiguousarray(np.concatenate([p["arrays"][k] for p in parts]))
    a["target"] = np.concatenate([p["arrays"]["target"] for p in parts])
    n = a["E"].size
    used = G - 1 if G > 2 else G
    a["group"] = np.floor(scenes.uniform(seed, 1, n) * (used + 1)).astype(np.int32) - 1
    th = [scenes.controller_params(seed, 10 + i, dim, G, K, H, sensor_gain=2.0) for i in range(len(sides))]
    a["w"] = np.stack(th).astype(np.float32)
    d.update(n_particles=[p["desc"]["n_particles"][0] for p in parts], n_scenes=len(sides), n_groups=G, n_basis=K,
             ctrl_hidden=H, ctrl_scale=20.0, act_period=17.0, ckpt_every=4)
    return s


@pytest.mark.parametrize("dim,G,K,H,sides", [(2, 1, 0, 1, (9,)), (2, 8, 8, 64, (24, 5)), (3, 3, 2, 33, (9, 4)), (3, 8, 0, 32, (16,)),
                                             (3, 5, 8, 63, (5, 12))])
def test_controller_shapes(mpm, dim, G, K, H, sides):
    scene, T = _scene(dim, G, K, H, sides), 10
    seeds = _random_seeds(scene, np.random.default_rng(7))
    g = _run_gpu(mpm, scene, T, seeds=seeds, loss=False)
    _compare_states(g["state"], _oracle_states(scene, T), scene, POS_TOL)
    o = _oracle_grad_linear(scene, T, {k: v.astype(np.float64) for k, v in seeds.items()})
    _compare_grads(g["grad"], o, KEYS)


def test_scene_alone_and_in_a_batch(mpm):
    scene, T = _scene(3, 4, 2, 16, (8, 12)), 8
    scene["desc"]["deterministic_p2g"] = 1
    whole = _run_gpu(mpm, scene, T, loss=False)["state"]
    for i in range(2):
        alone = _run_gpu(mpm, subset_scenes(scene, [i]), T, loss=False)["state"]
        for w, a in zip(whole, alone):
            assert np.array_equal(w[:, scene_slice(scene, i)], a)


def test_hidden_units_beyond_the_range(mpm):
    """A hidden unit's argument above FP32's range saturates it, as a smaller one of its sign does."""
    T = 8

    def run(w):
        scene = _scene(3, 2, 2, 8, (6, 5))
        scene["desc"].update(deterministic_p2g=1, act_phase=0.3)
        n_in = 2 + 2 * 3 * 2
        th = scene["arrays"]["w"].copy()
        for j in range(8):  # the time inputs' weights, one sign a unit
            th[:, j * n_in:j * n_in + 2] = w if j % 2 else -w
        scene["arrays"]["w"] = th
        seeds = _random_seeds(scene, np.random.default_rng(7))
        return _run_gpu(mpm, scene, T, seeds=seeds, loss=False)

    got, want = run(3e38), run(1e30)
    for a, b in zip(got["state"], want["state"]):
        assert np.isfinite(a).all() and np.array_equal(a, b)
    for key in got["grad"]:
        assert np.array_equal(got["grad"][key], want["grad"][key]), key
