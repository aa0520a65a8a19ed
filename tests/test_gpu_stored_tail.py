"""A forward pass that a backward is expected to follow stores its last two
checkpoint segments in the recomputation sets, and the backward starts with
their adjoint.  Every order of calls must give the oracle's gradients: the
first backward of a handle (recomputes everything), the following ones, a
second backward of the same forward, a forward that no backward followed, and
an option changed in between.  Tolerances as in test_gpu_parity.py."""
import functools

import numpy as np
import pytest

from paper_2503_22767_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22767_gb300 import binding as B  # noqa: E402
from paper_2503_22767_gb300.sim import Simulator  # noqa: E402

GRAD_COS, GRAD_REL = 0.999, 1e-3


def _t(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@functools.lru_cache(maxsize=None)
def _case(dim, segments):
    import oracle

    # a shear that carries particles across several cells, so that each
    # segment has its own particle order
    steps = 120
    every = -(-steps // segments)
    if dim == 2:
        w = W.walker_2d(seed=6, n_steps=steps, scale=0.3, checkpoint_every=every)
    else:
        w = W.walker_3d(seed=4, n_steps=steps, res=40, scale=0.2, checkpoint_every=every)
    w.v0 = np.zeros_like(w.x0)
    w.v0[0] = (8.0 if dim == 2 else 40.0) * (w.x0[1] - 0.3)
    return w, oracle.backward(w, ckpt_every=20)


def _check(sim, ob, n):
    got = dict(zip(("g_phi", "g_mag", "g_field"), sim.backward(torch.ones(n, device="cuda"))))
    for k, g in got.items():
        a, b = g.cpu().numpy().astype(np.float64).ravel(), np.asarray(ob[k], np.float64).ravel()
        na, nb = np.linalg.norm(a), np.linalg.norm(b)
        assert a @ b / (na * nb) >= GRAD_COS and np.linalg.norm(a - b) / nb <= GRAD_REL, k


MODES = {
    "default": {},
    "one_stream": {B.MPM_OPT_STREAMS: 1},
    "every_node": {B.MPM_OPT_GRID_BLOCKS: 0},
    "fused_grid": {B.MPM_OPT_FUSE_GRID: 3},
    "no_graphs": {B.MPM_OPT_GRAPHS: 0},
    "resident": {B.MPM_OPT_RESIDENT_SEGMENTS: 1},
}


@pytest.mark.parametrize("dim,segments", [(2, 1), (2, 2), (2, 3), (2, 5), (3, 1), (3, 2), (3, 4)])
@pytest.mark.parametrize("mode", list(MODES))
def test_every_order_of_calls(dim, segments, mode):
    w, ob = _case(dim, segments)
    n = w.cfg.n_instances
    sim = Simulator(w.cfg, options=MODES[mode])
    args = (_t(w.x0), _t(w.phi), _t(w.mag), _t(w.field))
    losses = []

    def forward():
        losses.append(float(sim.forward(*args, v0=_t(w.v0))[0]))

    forward()
    _check(sim, ob, n)       # nothing stored
    forward()
    _check(sim, ob, n)       # stored by the forward
    _check(sim, ob, n)       # consumed: recomputed
    forward()                # stored, but no backward follows
    forward()                # so this one does not store
    _check(sim, ob, n)
    forward()
    sim.set_option(B.MPM_OPT_ADJOINT_BLOCKS, 3 if dim == 2 else 2)  # an option changed: recomputed
    _check(sim, ob, n)
    forward()
    _check(sim, ob, n)
    np.testing.assert_allclose(losses, losses[0], rtol=1e-3)
    sim.close()
