"""The allocation-free substep leaves its accumulator zero for the next call
and keeps its error flags between calls in one word: a call must not depend on
the calls before it, whatever their dimension and grid, nor on an error they
reported.  Compared with the FP64 oracle at the parity tests' state
tolerance."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22767_gb300 import binding as B  # noqa: E402
from test_zz_no_alloc import CASES, STATE_TOL, _call, _config_c, _errors, _oracle_state, _t  # noqa: E402


@pytest.mark.parametrize("order", [("2d_floor", "3d_free", "2d_floor"), ("3d_free", "bad", "3d_free"),
                                   ("3d_free", "bad", "bad", "2d_floor", "3d_free")])
def test_a_call_does_not_depend_on_the_calls_before(order):
    lib = B.load()
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for key in order:
        w = CASES["2d_floor" if key == "bad" else key]()
        d, n = w.cfg.dim, w.cfg.n_total
        keep = []
        s0 = np.zeros((2 * d + 2 * d * d, n), np.float32)
        s0[:d] = w.x0
        if w.v0 is not None:
            s0[d:2 * d] = w.v0
        if key == "bad":
            s0[0, 0] = 1.5  # outside the grid (the kernels clamp the stencil)
        out = torch.empty((2 * d + 2 * d * d, n), device="cuda")
        torch.cuda.synchronize()
        st = _call(lib, _config_c(w.cfg, keep), 0, _t(s0), _t(w.phi), _t(w.mag), _t(w.field[0]), out, stream)
        if key == "bad":
            assert st == B.MPM_ERR_DOMAIN
            continue
        assert st == B.MPM_OK, lib.mpm_noalloc_last_error()
        errs = _errors(out.cpu().numpy().astype(np.float64), _oracle_state(w, 1), d, n)
        assert all(e <= STATE_TOL for e in errs.values()), errs
