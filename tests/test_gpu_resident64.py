"""Resident FP64 sweeps (one launch for many sweeps of a lattice that fits on the chip) are
bitwise the same number of one-sweep launches (a step of one sweep is one such launch), with
both pseudo-time steps and area multipliers, over brick cuts that are ragged in every
direction and from two to six cells per thread; transposed ones give the oracle's gradient."""
import functools

import numpy as np
import pytest

from oracle import soc
from tests._cases import problem_from_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_08034_gb300 import _build
    _build.build()


@functools.lru_cache(maxsize=None)
def _case(dims, seed=7):
    from paper_2502_08034_gb300 import synth
    return synth.build_case("res%dx%dx%d" % dims, dims, 0.82, 4.0, seed, 0.01, -0.10, 0.4, 1e-10,
                            flow_device="cuda")


@pytest.mark.parametrize("dims,sweeps", [((5, 7, 11), 9), ((24, 20, 37), 8), ((64, 40, 66), 5),
                                         ((61, 63, 64), 7), ((77, 60, 80), 4), ((72, 72, 88), 3)])
@pytest.mark.parametrize("dt_mode", ["local", "global"])
def test_resident_sweeps_are_bitwise_one_sweep_launches(dims, sweeps, dt_mode):
    from paper_2502_08034_gb300 import rfb, synth
    case = _case(dims)
    m = synth.lognormal_area_mult(case.solid)
    s0 = np.random.default_rng(3).random(case.n)
    out = []
    for steps in ([1] * sweeps, [sweeps]):
        with rfb.Solver.from_case(case, area_mult=m) as sv:
            sv.set_state(s0)
            l0 = sv.kernel_launches
            for n in steps:
                r = sv.step(case.s_in, case.eta, n, dt_mode=dt_mode)
            out.append((sv.get_state(), r["residual"], r["I_tot"], sv.kernel_launches - l0))
    assert out[1][3] < out[0][3]
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1:3] == out[1][1:3]


def test_more_sweeps_than_one_launch_takes():
    """2048 sweeps a launch; the next one starts from the state reached."""
    from paper_2502_08034_gb300 import rfb
    case = _case((24, 20, 37))
    out = []
    for steps in ((2047, 3), (2050,)):
        with rfb.Solver.from_case(case) as sv:
            for n in steps:
                sv.step(case.s_in, case.eta, n)
            out.append(sv.get_state())
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("objective", ["I_tot", "U_mt"])
def test_resident_adjoint_matches_the_oracle(objective):
    from paper_2502_08034_gb300 import rfb
    case = _case((21, 18, 33), 11)
    p = problem_from_case(case, soc)
    with rfb.Solver.from_case(case) as sv:
        sv.solve(case.s_in, case.eta, 1e-13)
        sv.umt(1e-13)
        dm, db, r = sv.adjoint(objective, 1e-13)
    ref = soc.adjoint(p, None, objective)
    scale = np.abs(ref["d_area_mult"]).max()
    assert np.abs(dm - ref["d_area_mult"]).max() <= 1e-9 * scale
    assert abs(db - ref["d_beta"]) <= 1e-9 * abs(ref["d_beta"])
