"""One step at the line lengths that no other step test reaches, against the
FP64 oracle: FP32 passes of 72, 144 and 288 points in x and in z, and the action
and observation transforms by lines of 8, 12, 48, 96 and 192 points, two and
eight lines per CTA.  Bars: those of the other step tests (all FP64 1e-11, mixed
1e-4).
"""

import pytest

from gpu_util import run_batch_pair
from test_gpu_dispatch_edges import _check

pytestmark = pytest.mark.gpu

# (nx, nz, batch): from 8192 points of a batch on the transforms go by lines;
# eight lines per CTA from 1216 lines of a pass on
SIZES = [(48, 96, 2), (96, 48, 2), (48, 96, 51), (96, 48, 51), (192, 8, 6), (8, 192, 6), (192, 8, 304), (8, 192, 304),
         (8, 12, 86), (12, 8, 86), (8, 12, 304), (12, 8, 304)]


@pytest.mark.parametrize("nx,nz,batch", SIZES)
@pytest.mark.parametrize("precision", [0, 1])
def test_step_line_lengths(native_gpu, nx, nz, batch, precision):
    kw = dict(nx=nx, ny=9, nz=nz, lx=2.67, lz=0.8, re_tau=180.0, re_bulk=2800.0, dt=0.002, precision=precision)
    _, res = run_batch_pair(native_gpu, kw, batch, [0, batch - 1], 1)
    _check(res, kw)
