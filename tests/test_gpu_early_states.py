"""Adjoint passes that read their state and form its stress before the pass ahead of them has ended:
the deterministic gradients are bitwise those of passes that each wait for the last (profiling launches
them one by one), with the re-simulation on the same stream or another, grids kept or recomputed, for
2D batches on both sides of the size up to which it is done, and materials that do and do not."""
import numpy as np
import pytest

from paper_1910_00935_gb300 import scenes
from test_gpu_parity import _random_seeds, mpm  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCENES = {
    "cube": lambda: scenes.make("cube3d", n_side=20, n_grid=64),
    "liquid": lambda: scenes.make("liquid3d", cols=(12, 20, 9)),
    "robots": lambda: scenes.make("robots3d", n_scenes=2, dims=(12, 8, 8)),
    "square": lambda: scenes.make("square2d", n_side=45),
    "2D, below two waves": lambda: scenes.make("rects2d", n_scenes=20, n_min=9500, n_max=9500),
    "2D, above two waves": lambda: scenes.make("rects2d", n_scenes=20, n_min=10000, n_max=10000),
}


@pytest.mark.parametrize("name", list(SCENES))
def test_equals_passes_one_by_one(mpm, name):  # noqa: F811
    scene, T = SCENES[name](), 11
    scene["desc"]["deterministic_p2g"], scene["desc"]["ckpt_every"] = 1, 4
    seeds = {k: torch.as_tensor(v).cuda() for k, v in _random_seeds(scene, np.random.default_rng(2)).items()}

    def grads(**options):
        sim = mpm.from_scene(scene, max_steps=T)
        for k, v in options.items():
            sim.set_option(getattr(mpm, "MPM_OPT_" + k), v)
        sim.forward(T)
        out = [t.clone() for t in sim.backward(**seeds).values()]
        sim.check()
        sim.close()
        return out

    want = grads(PROFILE=1)
    for options in ({}, {"USE_GRAPHS": 0}, {"OVERLAP_RESIM": 0}, {"GRID_RECOMPUTE": 1}, {"GRID_RECOMPUTE": 1, "OVERLAP_RESIM": 0}):
        assert all(torch.equal(a, b) for a, b in zip(grads(**options), want)), options


@pytest.mark.parametrize("name", list(SCENES))
def test_equals_passes_one_by_one_without_gather_box(mpm, name):  # noqa: F811
    """Without the shared gather box a pass's grid reads hang on nothing but its particles' positions,
    which an early pass has before the grid is written."""
    scene, T = SCENES[name](), 7
    scene["desc"]["deterministic_p2g"], scene["desc"]["ckpt_every"] = 1, 4
    seeds = {k: torch.as_tensor(v).cuda() for k, v in _random_seeds(scene, np.random.default_rng(2)).items()}

    def run(profile):
        sim = mpm.from_scene(scene, max_steps=T)
        sim.set_option(mpm.MPM_OPT_PROFILE, profile)
        sim.set_option(mpm.MPM_OPT_GATHER_CAPACITY, 0)
        sim.forward(T)
        out = [t.clone() for t in sim.state()] + [t.clone() for t in sim.backward(**seeds).values()]
        sim.check()
        sim.close()
        return out

    assert all(torch.equal(a, b) for a, b in zip(run(0), run(1)))
