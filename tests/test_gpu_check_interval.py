"""Check intervals of default mixed solves: whole multiples of the sweeps of the launches that a
lattice's resident sweeps replaced (one, two or three), so a solve stops at the sweep, with the
bits, of a solve by those launches; beyond the chip it stops like one of the three."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEPTH = {1: "plain", 2: "blocked_chunked", 3: "three_sweep_chunked"}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_08034_gb300 import _build
    _build.build()


@functools.lru_cache(maxsize=None)
def _case(dims):
    from paper_2502_08034_gb300 import synth
    return synth.build_case("ci%dx%dx%d" % dims, dims, 0.82, 6.0, 5, 0.01, -0.10, 0.4, 1e-10,
                            flow_device="cuda", flow_tol=1e-10)


def _solves(dims, kernel):
    """(sweeps, field) at several tolerances and operating points, each from a cold start."""
    from paper_2502_08034_gb300 import rfb
    case, out = _case(dims), []
    with rfb.Solver.from_case(case) as sv:
        for eta, tol in ((-0.10, 1e-8), (-0.06, 3e-9), (-0.03, 1e-9), (-0.12, 3e-10),
                         (-0.08, 1e-10)):
            sv.reset_state()
            r = sv.solve(case.s_in, eta, tol, precision="mixed", fp32_kernel=kernel)
            out.append((r["sweeps"], sv.get_state()))
        u, r = sv.umt(1e-9, precision="mixed", fp32_kernel=kernel)
        out.append((r["sweeps"], np.array(u)))
    return out


# one wave of one-sweep blocks; more, whose two-sweep launches were the faster; three-sweep ones
@pytest.mark.parametrize("dims,depth", [((64, 64, 64), 1), ((88, 84, 110), 1), ((24, 203, 63), 1),
                                        ((32, 81, 165), 2), ((72, 64, 176), 2),
                                        ((132, 44, 114), 3), ((136, 76, 69), 3),
                                        ((64, 88, 141), 3)])
def test_resident_solves_stop_like_the_launches_they_replaced(dims, depth):
    got, want = _solves(dims, "resident"), _solves(dims, DEPTH[depth])
    assert [n for n, _ in _solves(dims, "auto")] == [n for n, _ in got]
    assert [n for n, _ in got] == [n for n, _ in want]
    for (_, s), (_, t) in zip(got, want):
        assert np.array_equal(s, t)


@pytest.mark.parametrize("dims", [(164, 100, 70), (256, 61, 86)])
def test_solves_beyond_the_chip_stop_like_one_of_the_depths(dims):
    got = _solves(dims, "auto")
    want = {d: _solves(dims, k) for d, k in DEPTH.items()}
    like = [d for d, w in want.items() if [n for n, _ in w] == [n for n, _ in got]]
    assert like
    for (_, s), (_, t) in zip(got, want[like[0]]):
        assert np.array_equal(s, t)
