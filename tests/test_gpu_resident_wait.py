"""Failure detection of the resident kernels, without a fault: a wait that gives up (after one
poll, when its words are still on their way) ends the call with an error at that cycle, whichever
call it is, and the calls after it return what a fresh handle returns."""
import dataclasses
import functools
import time

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
def _case():
    from paper_2502_08034_gb300 import synth
    return synth.build_case("wait", (36, 32, 40), 0.82, 4.0, 3, 0.01, -0.10, 0.4, 1e-10)


def _refused(sv, call):
    """The call ends with RFB_ERR_CUDA, at once, when waits give up after one poll."""
    from paper_2502_08034_gb300 import rfb
    sv.selftest_wait_limit(1)
    t0 = time.monotonic()
    with pytest.raises(rfb.RfbError) as e:
        call()
    assert e.value.status == rfb.RFB_ERR_CUDA and "waited too long" in str(e.value)
    assert time.monotonic() - t0 < 20
    sv.selftest_wait_limit(0)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_adjoint_stops_at_the_cycle(precision):
    from paper_2502_08034_gb300 import rfb
    case, out = _case(), []
    for fail in (True, False):
        with rfb.Solver.from_case(case) as sv:
            sv.solve(case.s_in, case.eta, 1e-12)
            if fail:
                # 400 sweeps a cycle: without a stop at the first the call would take hours
                _refused(sv, lambda: sv.adjoint("I_tot", 1e-30, precision=precision,
                                                check_every=400))
            dm, db, r = sv.adjoint("I_tot", 1e-11, precision=precision)
            out.append((dm, db, r["sweeps"]))
    assert out[0][1:] == out[1][1:] and np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solves_stop_at_the_cycle(precision):
    from paper_2502_08034_gb300 import rfb
    case, out = _case(), []
    for fail in (True, False):
        with rfb.Solver.from_case(case) as sv:
            if fail:
                _refused(sv, lambda: sv.solve(case.s_in, case.eta, 1e-30, precision=precision))
                _refused(sv, lambda: sv.umt(1e-30, precision=precision))
                _refused(sv, lambda: sv.step(case.s_in, case.eta, 500, precision=precision))
                sv.reset_state()
            r = sv.solve(case.s_in, case.eta, 1e-10, precision=precision)
            u, _ = sv.umt(1e-10, precision=precision)
            out.append((r["I_tot"], u, r["sweeps"], sv.get_state()))
    assert out[0][:3] == out[1][:3] and np.array_equal(out[0][3], out[1][3])


def test_potential_solves_after_one_that_gave_up():
    """Blocks that went on after the first one had given up leave words with tags that the next
    solve uses: it must not take them (solves cut off at many points, then one to its end)."""
    from paper_2502_08034_gb300 import rfb, synth
    case = dataclasses.replace(synth.build_case("waitbv", (13, 11, 15), 0.82, 4.0, 5, 0.002, -0.10,
                                                0.2, 1e-12, flow_device="cuda"), k0=2e-5)
    out = []
    for fail in (True, False):
        with rfb.Solver.from_case(case) as sv:
            sv.solve(case.s_in, case.eta, 1e-12)
            kw = dict(start="sbv", cycle=50, max_sweeps=100, allow_not_converged=True)
            for polls in range(1, 13) if fail else ():
                sv.selftest_wait_limit(polls)
                try:
                    sv.solve_bv(case.s_in, case.eta, 1e-30, **kw)
                    assert polls > 1
                except rfb.RfbError as e:
                    assert e.status == rfb.RFB_ERR_CUDA
                sv.selftest_wait_limit(0)
            r = sv.solve_bv(case.s_in, case.eta, 1e-30, **kw)
            out.append((r["I_tot"], r["cg_iterations"], r["phi_min"], sv.get_bv_state()))
    assert out[0][:3] == out[1][:3]
    for k, x in out[0][3].items():
        assert np.array_equal(x, out[1][3][k])


def test_wait_limit_arguments():
    from paper_2502_08034_gb300 import rfb
    with rfb.Solver.from_case(_case()) as sv:
        for bad in (-1, (1 << 26) + 1):
            with pytest.raises(rfb.RfbError) as e:
                sv.selftest_wait_limit(bad)
            assert e.value.status == rfb.RFB_ERR_INVALID_ARG
