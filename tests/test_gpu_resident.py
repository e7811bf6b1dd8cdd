"""Resident FP32 sweeps (a lattice that fits on the chip, one launch for the sweeps of a
correction cycle) are bitwise the same number of one-sweep launches, forward and transposed,
with area multipliers and pinned cells, over brick cuts that are ragged in every direction,
one brick across, a few cells per thread and the most that fit; widths that are no multiple
of 4 (whose one-sweep kernel rounds differently) reach the oracle's steady state."""
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


@pytest.mark.parametrize("dims,sweeps", [((8, 8, 12), (1, 2, 3)), ((24, 20, 37), (7, 200)),
                                         ((64, 64, 64), (50, 1)), ((100, 12, 90), (33, 34)),
                                         ((12, 150, 50), (40,)), ((16, 16, 32), (4097, 8200)),
                                         ((88, 84, 110), (25, 60))])
def test_resident_sweeps_are_bitwise_one_sweep_launches(dims, sweeps):
    """Also cycles longer than one launch (4096 sweeps), whose next launch starts from the
    correction reached so far."""
    from paper_2502_08034_gb300 import rfb, synth
    case = _case(dims)
    m = synth.lognormal_area_mult(case.solid)
    states = []
    for kernel in ("plain", "auto"):
        with rfb.Solver.from_case(case, area_mult=m) as sv:
            for n in sweeps:
                sv.step(case.s_in, case.eta, n, precision="mixed", fp32_kernel=kernel)
            states.append(sv.get_state())
            if kernel == "auto":
                assert sv.tuned_fp32_kernel()[0] == "resident"
    assert np.array_equal(states[0], states[1])


def test_resident_transposed_sweeps_and_umt():
    """The adjoint with and without a pass variant chosen before, and U_mt with its pinned
    cells, against the launches they replace."""
    from paper_2502_08034_gb300 import rfb, synth
    case = _case((52, 44, 30))
    m = synth.lognormal_area_mult(case.solid)
    out = []
    for kernel in ("blocked_chunked", "auto"):
        with rfb.Solver.from_case(case, area_mult=m) as sv:
            r = sv.solve(case.s_in, case.eta, 1e-10, precision="mixed", fp32_kernel=kernel,
                         check_every=100)
            u, _ = sv.umt(1e-10, precision="mixed", fp32_kernel=kernel, check_every=100)
            dm, db, a = sv.adjoint("I_tot", 1e-11, precision="mixed", check_every=100)
            out.append((r["I_tot"], u, dm, db, a["sweeps"]))
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("dims", [(5, 7, 11), (33, 18, 41)])
def test_resident_solve_of_any_width_matches_the_oracle(dims):
    from paper_2502_08034_gb300 import rfb
    case = _case(dims, 11)
    ref = soc.steady_state(soc.assemble(problem_from_case(case, soc)))
    with rfb.Solver.from_case(case) as sv:
        r = sv.solve(case.s_in, case.eta, 1e-11, precision="mixed")
        s = sv.get_state()
        assert sv.tuned_fp32_kernel()[0] == "resident"
    assert r["residual"] <= 1e-11
    assert np.abs(s - ref).max() < 1e-7


def test_a_lattice_beyond_the_chip_is_timed_as_before():
    from paper_2502_08034_gb300 import rfb
    case = _case((128, 96, 96))
    with rfb.Solver.from_case(case) as sv:
        sv.solve(case.s_in, case.eta, 1e-6, precision="mixed")
        assert sv.tuned_fp32_kernel()[0] != "resident"
