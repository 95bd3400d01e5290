"""Film right-hand sides where the transform core changes its shape: every elements-per-thread choice
per axis and precision, lines shorter and longer than a warp, non-square grids whose axes take
different ones, ragged conductors with a filled hole, and the checkpoint's row-major warm start."""
import ctypes

import numpy as np
import pytest

import workloads as W
from helpers import oracle_of, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1801_04869_gb300 import native  # noqa: E402

# FP64: the transform's rounding (1e-16 relative, a few thousand of them amplified by the smoothed
# derivatives) is far below 1e-9; FP32: the same with 6e-8 stays below 2e-4
TOL = {0: 1e-9, 1: 2e-4}


def _film(nx, ny, precision):
    """A ragged film of about half the box with a filled hole and a jc map."""
    Lx, Ly = 2.0 * nx / max(nx, ny), 2.0 * ny / max(nx, ny)
    m = W.film_mask(nx, ny, Lx, Ly, "rect", ax=0.53 * Lx, ay=0.47 * Ly, cx=0.03 * Lx,
                    hole=(0.1 * Lx, 0.0, 0.2 * min(Lx, Ly)))
    wl = W.Workload(f"film_{nx}x{ny}", 2, nx, ny, 1, Lx, Ly, 0.0, m, n=19.0, rho_out=1.0,
                    precision=precision, t0=0.0, t1=1.0, he_knots=((0.0, 1.0), (0.0, 0.5)))
    wl.jc_map = W.jc_map_lognormal((ny, nx), seed=11)
    return wl


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(8, 8), (16, 8), (8, 32), (64, 16), (32, 128), (256, 256),
                                   (512, 128), (128, 512), (512, 256), (1024, 32), (1024, 1024),
                                   (2048, 8), (8, 2048), (2048, 512), (512, 2048)])
def test_rhs_matches_oracle(nx, ny, precision):
    wl = _film(nx, ny, precision)
    p, o = native.from_workload(wl), oracle_of(wl)
    g = W.film_state(wl.mask, wl.Lx, wl.Ly, seed=7, amplitude=0.4)
    y = torch.as_tensor(g, device="cuda")
    out = torch.zeros_like(y)
    for k in (1, 3):                     # a cold call, then one from its warm start
        ref, it_o, st_o = o.rhs(0.25, g, None, k)
        it_g, _ = p.mf_rhs(0.25, y, out, force_iters=k, allow_noconv=True)
        assert it_g == it_o == k
        assert rel_l2(out.cpu().numpy(), ref) < TOL[precision]


@pytest.mark.parametrize("precision", [0, 1])
def test_checkpoint_keeps_the_warm_start_row_major(precision):
    """The h_dot iterate lies in the blob behind the header (48 bytes), the solver state and the six
    FP64 buffers, row-major in the transform precision, whatever layout the kernels use."""
    wl = _film(64, 32, precision)
    p, o = native.from_workload(wl), oracle_of(wl)
    g = W.film_state(wl.mask, wl.Lx, wl.Ly, seed=7, amplitude=0.4)
    y = torch.as_tensor(g, device="cuda")
    p.mf_rhs(0.25, y, torch.zeros_like(y), force_iters=3, allow_noconv=True)
    o.rhs(0.25, g, None, 3)
    blob = p.mf_checkpoint_save().cpu().numpy()
    n, ts = wl.nx * wl.ny, 4 if precision else 8
    log = 65536 * ctypes.sizeof(native.mf_step_log)      # the step log ends the blob
    hd = blob[blob.size - log - 2 * n * ts:][:n * ts].view(np.float32 if precision else np.float64)
    A = blob[48 + 16:48 + 24].view(np.float64)[0]        # the shift still to subtract
    got = hd.reshape(wl.ny, wl.nx).astype(np.float64) - A
    free = wl.mask == 0
    assert rel_l2(got[free], o.warm[free]) < TOL[precision]
