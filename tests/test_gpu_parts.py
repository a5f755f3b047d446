"""The mixed kernels' parts (N = 1,024, N = 512, N <= 256) chained in one call:
a candidate's results do not depend on what else the call holds, so every
window must get the same bits alone as beside windows of the other parts.
Candidate counts give items of one, an odd number and the most candidates."""
import pytest
import torch

from paper_2307_03763_gb300 import api
from paper_2307_03763_gb300 import workloads as wk

from tests.test_gpu_tchannel import _c, _problem

pytestmark = pytest.mark.gpu

SPECS = [(16e-3, 1024), (4e-3, 256), (11e-3, 512), (2e-3, 128), (15e-3, 1024), (1e-3, 64), (0.4e-3, 32), (9e-3, 512)]


@pytest.mark.parametrize("name", ["loglik", "loglik_aet", "loglik_phase", "loglik_phase_aet", "loglik_grad",
                                  "loglik_grad_aet"])
@pytest.mark.parametrize("n", [1, 33, 1500, 6001])
def test_parts_do_not_interact(name, n):
    ctx = api.Context(wk.YEAR)
    wins, th, data, weights = _problem(n, SPECS, n)
    d, w, th = [_c(x, torch.complex128) for x in data], [_c(x, torch.float64) for x in weights], _c(th, torch.float64)
    if not name.endswith("_aet"):
        d, w = d[:2], w[:2]
    call = getattr(ctx, name)
    joint = [x.clone() for x in call(wins, *d, *w, th, prec="mixed")]
    for k0, W, N, off, coff, m in wins:
        rows, bins = slice(coff, coff + m), slice(off, off + W)
        alone = call([(k0, W, N, 0, 0, m)], *[x[bins].clone() for x in d], *[x[bins].clone() for x in w],
                     th[rows].clone(), prec="mixed")
        for a, b in zip(joint, alone):
            assert torch.isfinite(b).all() and torch.equal(a[rows], b)
