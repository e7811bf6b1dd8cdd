"""One handle solved with local steps and then with the global one: the pass chosen (or asked
for) with local steps says nothing about the global step, whose passes take fewer lattices (nx a
multiple of 16, no area multipliers) and two sweeps each. The same bits as a fresh handle."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_08034_gb300 import _build
    _build.build()


@functools.lru_cache(maxsize=None)
def _case(dims):
    from paper_2502_08034_gb300 import synth
    return synth.build_case("sm%dx%dx%d" % dims, dims, 0.82, 6.0, 3, 0.01, -0.10, 0.4, 1e-10,
                            flow_device="cuda", flow_tol=1e-10)


# (nx % 16 != 0: no pass of the global step; nx % 16 == 0: none with multipliers, else its own)
@pytest.mark.parametrize("dims", [(164, 100, 70), (176, 90, 80)])
@pytest.mark.parametrize("mult", ["", "at first", "between"])
@pytest.mark.parametrize("first", ["auto", "blocked", "three_sweep_chunked"])
def test_local_steps_then_the_global_step(dims, mult, first):
    from paper_2502_08034_gb300 import rfb, synth
    case = _case(dims)
    m = synth.lognormal_area_mult(case.solid) if mult else None
    out = []
    for before in (True, False):
        with rfb.Solver.from_case(case, area_mult=m if mult == "at first" else None) as sv:
            if before:
                sv.step(case.s_in, case.eta, 12, precision="mixed", fp32_kernel=first)
                sv.reset_state()
            if mult == "between":
                sv.set_area_mult(m)
            for n in (7, 12):
                r = sv.step(case.s_in, case.eta, n, precision="mixed", dt_mode="global")
            out.append((r["residual"], sv.get_state()))
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])


def test_multipliers_after_a_global_solve():
    from paper_2502_08034_gb300 import rfb, synth
    case = _case((176, 90, 80))
    m = synth.lognormal_area_mult(case.solid)
    out = []
    for before in (True, False):
        with rfb.Solver.from_case(case) as sv:
            if before:
                sv.step(case.s_in, case.eta, 12, precision="mixed", dt_mode="global")
                sv.reset_state()
            sv.set_area_mult(m)
            sv.step(case.s_in, case.eta, 9, precision="mixed", dt_mode="global")
            out.append(sv.get_state())
    assert np.array_equal(out[0], out[1])
