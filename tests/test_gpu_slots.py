"""Sums over all particles of an instance (momentum rows of the locomotion
objective, dL/dB_applied, dL/dG) are added in 64 bits to 1 .. 16 slots per
instance and substep and folded at the end of the pass.  Around the sizes
where the slot count changes, with instances that share warps, against the
FP64 oracle.  Tolerances as in test_gpu_parity.py."""
import numpy as np
import pytest

from paper_2503_22767_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22767_gb300.sim import Simulator  # noqa: E402


def _t(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _body(cells, seed):
    return W.tiny_2d(seed=seed, n_steps=10, res=96, cells=cells, bound=3, lift=3, loss_kind=1, wall_mode=1, phi_lo=0.3,
                     gravity=-9.81, field_scale=0.2, mag_scale=1.0, v_scale=0.2)


# slots: 1, 1, 2, 8, 16, and 4 over four uneven instances (1,024 particles per slot)
@pytest.mark.parametrize("bodies", [[(7, 57)], [(7, 57), (16, 32)], [(16, 32)], [(50, 55)], [(80, 52)],
                                    [(3, 3), (50, 50), (5, 1), (40, 41)]])
@pytest.mark.parametrize("gradient", [False, True])
def test_slots_match_oracle(bodies, gradient):
    import oracle

    parts = [_body(c, 31 + i) for i, c in enumerate(bodies)]
    w = W.batch(parts) if len(parts) > 1 else parts[0]
    rng = np.random.default_rng(5)
    if gradient:
        w.fgrad = (0.5 * rng.uniform(-1, 1, size=(w.cfg.n_instances, w.cfg.n_steps, 2, 2))).astype(np.float32)
    of, ob = oracle.forward(w), oracle.backward(w)
    sim = Simulator(w.cfg)
    if gradient:
        sim.set_field_gradient(_t(w.fgrad))
    loss, _ = sim.forward(_t(w.x0), _t(w.phi), _t(w.mag), _t(w.field), v0=_t(w.v0))
    # the objective is a mean velocity whose terms (random v0) nearly cancel:
    # each of the 10 substeps rounds a velocity by a few 2^-24 of its size
    terms = w.cfg.n_steps * w.cfg.dt * np.abs(w.v0[0]).mean()
    np.testing.assert_allclose(loss.cpu().numpy(), of["loss"], rtol=1e-5, atol=40 * 2.0 ** -24 * terms)
    out = dict(zip(("g_phi", "g_mag", "g_field"), sim.backward(torch.ones(w.cfg.n_instances, device="cuda"))))
    if gradient:
        out["g_fgrad"] = sim.field_gradient_grad()
    for k, g in out.items():
        a, b = g.cpu().numpy().astype(np.float64), np.asarray(ob[k], np.float64)
        assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b), k
    sim.close()
