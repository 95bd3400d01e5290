"""Bulk right-hand sides where the passes change their shape: every elements-per-thread choice per axis
and precision, the smallest and longest lines, x items of one to many row units, z groups of one to
four lines, under the elliptic and field-dependent laws with a jc map."""
import numpy as np
import pytest

import workloads as W
from helpers import oracle_of, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1801_04869_gb300 import native  # noqa: E402

# as for the film's shapes: rounding amplified by the law (n = 19) and the smoothed derivatives
TOL = {0: 1e-9, 1: 2e-4}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dims", [(8, 8, 8), (512, 8, 8), (8, 512, 8), (8, 8, 512), (32, 16, 8),
                                  (16, 128, 64), (64, 64, 32), (64, 64, 64), (128, 64, 64),
                                  (256, 64, 8), (256, 256, 64)])
def test_rhs_matches_oracle(dims, precision):
    nx, ny, nz = dims
    L = tuple(2.0 * n / max(dims) for n in dims)
    m = W.bulk_mask(nx, ny, nz, *L, "box", ax=0.5 * L[0], ay=0.5 * L[1], az=0.5 * L[2])
    wl = W.Workload(f"bulk_{nx}x{ny}x{nz}", 3, nx, ny, nz, *L, m, n=19.0, rho_out=5.0, precision=precision,
                    t0=0.0, t1=1.0, he_knots=((0.0, 0.5, 1.0), (0.0, 0.25, 0.25)), gamma=1.5, b0=0.4,
                    vector_he=(0.3, 0.0, 1.0))
    wl.jc_map = W.jc_map_lognormal((nz, ny, nx), seed=11)
    h = W.bulk_state(wl.mask, L, seed=7, h0=0.3, depth=0.3)
    p, o = native.from_workload(wl), oracle_of(wl)
    y = torch.as_tensor(np.ascontiguousarray(h), device="cuda")
    out = torch.zeros_like(y)
    for k in (1, 2):                     # a cold call, then one from its warm start
        ref, it_o, _ = o.rhs(0.25, h, None, k)
        it_g, _ = p.mf_rhs(0.25, y, out, force_iters=k, allow_noconv=True)
        assert it_g == it_o == k
        assert rel_l2(out.cpu().numpy(), ref) < TOL[precision]
