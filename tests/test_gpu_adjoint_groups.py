"""The actuation's gradient where the particles of one warp belong to many groups or to one, with tiles
that end inside a warp, and the adjoint's two ways of holding its carried values (grids kept, grids
recomputed), against the FP64 oracle at the gradients' bar."""
import numpy as np
import pytest

from paper_1910_00935_gb300 import scenes
from test_gpu_parity import _compare_grads, _oracle_grad_linear, _random_seeds, _run_gpu, mpm  # noqa: F401

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recompute", [0, 1])
@pytest.mark.parametrize("spread", ["every lane another", "one group", "last particle alone"])
def test_groups_of_a_warp(mpm, spread, recompute):  # noqa: F811
    scene = scenes.make("robots3d", n_scenes=2, dims=(13, 7, 9))
    N, G, rng = sum(scene["desc"]["n_particles"]), scene["desc"]["n_groups"], np.random.default_rng(11)
    scene["arrays"]["group"][:] = {"every lane another": np.arange(N) % G, "one group": np.full(N, G - 1),
                                   "last particle alone": np.where(np.arange(N) == N - 1, 0, 1)}[spread]
    scene["desc"]["ckpt_every"] = 3
    seeds = _random_seeds(scene, rng)
    got = _run_gpu(mpm, scene, 7, seeds, loss=False, options={mpm.MPM_OPT_GRID_RECOMPUTE: recompute})
    want = _oracle_grad_linear(scene, 7, {key: v.astype(np.float64) for key, v in seeds.items()})
    _compare_grads(got["grad"], want, ("gx0", "gv0", "gC0", "gF0", "gw"))
