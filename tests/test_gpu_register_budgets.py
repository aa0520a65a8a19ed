"""The 3D particle kernels pick a register budget by the launch: 128 registers
for a body that one wave of the GPU holds (16 warps of 32 particles per SM),
past it 96 in blocks of up to 128 threads and 80 in larger ones.  Just below
and above that size, with and without the rules' other kernels (block sizes,
the option's budgets), the states and gradients must agree with one another
at float32 rounding; against the FP64 oracle the sizes below are covered by
test_gpu_parity.py."""
import numpy as np
import pytest

from paper_2503_22767_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22767_gb300 import binding as B  # noqa: E402
from paper_2503_22767_gb300.sim import Simulator  # noqa: E402


def _t(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _run(w, options):
    sim = Simulator(w.cfg, options=options)
    sim.forward(_t(w.x0), _t(w.phi), _t(w.mag), _t(w.field), target=_t(w.target))
    u, v, _, E = sim.read_state_strain()
    out = (u, v, E) + tuple(sim.backward(torch.ones(w.cfg.n_instances, device="cuda")))
    sim.close()
    return [t.double().cpu().numpy() for t in out]


# position errors grow by a few 2^-24 of the motion per substep: 10 substeps,
# and the gradients' sums over a hundred thousand particles
REL = 1e-4


@pytest.mark.parametrize("side", ["below", "at", "above"])
def test_budgets_agree_around_one_wave(side):
    wave = 512 * torch.cuda.get_device_properties(0).multi_processor_count
    # layers of 16 x 16 cells x 8 particles, the ragged end cut off the arrays
    n = {"below": wave - 1, "at": wave, "above": wave + 1}[side]
    depth = -(-n // (8 * 16 * 16))
    full = W.plate_3d(seed=3, n_steps=10, res=64, n_tasks=1, cells=(depth, 16, 16))
    cfg = W.MpmConfig(**{**full.cfg.as_dict(), "counts": [n], "checkpoint_every": 5})
    w = W.Workload("cut", cfg, full.x0[:, :n], None, full.phi[:n], full.mag[:, :n], full.field, full.target[:, :n])
    ref = _run(w, {})
    for options in ({B.MPM_OPT_BLOCK: 256}, {B.MPM_OPT_BLOCK: 64}, {B.MPM_OPT_ADJOINT_BLOCKS: 2}):
        for a, b in zip(_run(w, options), ref):
            assert np.linalg.norm(a - b) <= REL * np.linalg.norm(b), options
