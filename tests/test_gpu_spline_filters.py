"""Spline coefficients of grids that take the warmed-up filters.

The chunks start from a carry that is off by (2 - sqrt(3))^32 = 5e-19 of the
largest coefficient, and each sweep rounds once or twice per entry with a factor
1 / (1 - 0.27); two axes, against an oracle whose sweeps round as much: a few
tens of 2^-53 of the largest coefficient, 1e-14; in FP32 of 2^-24, 5e-6.
"""
import numpy as np
import pytest

import oracle.oracle as O
from paper_1705_03750_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1705_03750_gb300 import build as B  # noqa: E402

B.build()
from paper_1705_03750_gb300 import vlamet as V  # noqa: E402


# rows: chunks of 2 to 128 entries, one segment up to 4096, several beyond;
# columns: one block of up to 320 rows, one row more, the next blocks' edges;
# the shortest sides that the filters take, and shorter ones
@pytest.mark.parametrize("nx,nv", [(182, 181), (320, 110), (321, 105), (640, 53), (641, 52), (1030, 33), (993, 33),
                                   (33, 993), (9000, 4), (4, 8200), (36, 4096), (37, 4097), (34, 8192), (33, 8193),
                                   (1000, 32), (64, 1024), (33, 1057), (1300, 3000)])
@pytest.mark.parametrize("prec,scale", [("fp64", 1.0), ("fp64", 1e-280), ("fp32", 1.0), ("fp32", 1e-20)])
def test_coefficients_match_the_oracles(nx, nv, prec, scale):
    rc = I.SPITZER_128.with_(nx=nx, nv=nv, s=4)
    f0 = scale * np.random.default_rng(nx + nv).standard_normal((nx, nv))
    if prec == "fp32":
        f0 = f0.astype(np.float32).astype(np.float64)
    g = V.Solver(V.Config.from_run(rc, V.VM_FP64 if prec == "fp64" else V.VM_FP32_MIXED))
    g.set_f(f0)
    ref = O.spline_solve_2d(f0)
    tol = 1e-14 if prec == "fp64" else 5e-6
    assert np.abs(g.read_eta() - ref).max() <= tol * np.abs(ref).max()
