"""The mixed kernels' generated strain on both sides of the rotation's limit (rotated within a window, or sample by
sample where the frequency drifts too fast) against the oracle on the exact polarisations (binary128, rounded
once).  At 0.1 mHz TDI cancels the strain by ~1e5, so the mixed tolerance of 1e-6 sees errors of 1e-11 in it."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2204_06633_gb300 as lr  # noqa: E402
import synth  # noqa: E402
from _gpu import Pair, assert_close, host  # noqa: E402

if not oracle.quad_available():
    pytest.skip("no binary128 libm in this toolchain", allow_module_level=True)


@pytest.mark.parametrize("dt", [10.0, 7.25])
@pytest.mark.parametrize("f,fdot,fddot", [(1e-4, 0.0, 0.0), (1e-4, 1e-17, 0.0), (1e-4, -5e-16, 0.0), (1e-4, 1e-14, 0.0),
                                          (1.5e-4, 1e-16, 1e-25), (1e-4, 1e-16, 1e-28)])
def test_generated_strain_against_oracle(dt, f, fdot, fddot):
    N, p, t0 = 3000, 25, 1.0e7
    pair = Pair(lr.Context(0), synth.orbit_flexing(t0 - 3e5, t0 + N * dt + 3e5))
    src = dataclasses.replace(synth.draw_sources(1, seed=5)[0], f=f)
    gb = (src.A, f, fdot, fddot, src.phi0, src.iota)
    sky = (src.lam, src.beta, src.psi)
    plan = lr.Plan(pair.gpu.ctx, p, N, dt, pair.gpu, t0=t0, precision=lr.MIXED)
    got = host(plan.response_gb(gb, sky))
    plan.check()
    m = synth.input_margin_samples(dt, p)
    t0h = t0 - m * dt
    hp, hc = oracle.gb_polarisations(*gb, t0h, dt, N + 2 * m, quad=True)
    args = (p, 2, dt, t0, N, pair.orc, pair.orc, hp, hc, t0h, *sky)
    assert_close(got, oracle.response(*args), oracle.response(*args, absval=True), p + 1, 1e-6)
