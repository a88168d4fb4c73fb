"""The mixed fused kernel with 512 threads (launches of at most one tile per SM) against the one with 256: the
work items are the same, so the outputs are, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2204_06633_gb300 as lr  # noqa: E402
import synth  # noqa: E402
from _gpu import DT, T0, dev, host, run_case, Pair, sky  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    return lr.Context(0)


@pytest.mark.parametrize("p", [1, 7, 15, 25, 31])
@pytest.mark.parametrize("gen,mode", [(1, lr.DELAY_SUM), (2, lr.DELAY_SUM), (2, lr.DELAY_NESTED)])
def test_wide_equals_narrow(ctx, p, gen, mode):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    orb = synth.orbit_flexing(T0 - 3e5, 1e6)
    o = lr.Orbit(ctx, orb.t_knots, orb.pos, None)
    src = synth.draw_sources(1, seed=p)[0]
    tile = lr.Plan(ctx, p, 1, DT, o, t0=T0, precision=lr.MIXED).tile
    n_wide, n_narrow = sms * tile, (sms + 20) * tile + 7   # the last length of one wave, and more than one
    t0h, hp, hc = synth.gb_input(src, T0, DT, n_narrow, p)
    out = []
    for n in (n_wide, n_narrow):
        plan = lr.Plan(ctx, p, n, DT, o, t0=T0, precision=lr.MIXED, generation=gen, delay_mode=mode)
        out.append(host(plan.response(dev(hp), dev(hc), t0h, sky(src))))
        plan.check()
        last = plan.valid_range()[1]
        if n == n_wide:
            valid = last
    np.testing.assert_array_equal(out[0][:, :valid], out[1][:, :valid])


@pytest.mark.parametrize("N", [1, 3, 339, 340, 341, 4096])
def test_wide_small_lengths(ctx, N):
    run_case(ctx, synth.draw_sources(1, seed=N)[0], N, 25, Pair(ctx, synth.orbit_flexing(-2e6, 2e6)), precision=lr.MIXED,
             rel=1e-6)
