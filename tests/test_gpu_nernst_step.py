"""The fused Nernst step (electrode cells by 64 from their list, the rest in 32 x 2 x 2 tiles) at
ragged tile edges in every direction, with area multipliers: the oracle's SBV steady state at
the bar of the model's other tests (1e-10 relative)."""
import dataclasses

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


@pytest.mark.parametrize("dims", [(33, 7, 9), (31, 10, 16), (66, 9, 11)])
def test_fused_step_reaches_the_oracle(dims):
    from paper_2502_08034_gb300 import rfb, synth
    c = synth.build_case("ns%dx%dx%d" % dims, dims, 0.85, 3.0, 21, 0.01, -0.10, 0.5, 1e-12)
    c = dataclasses.replace(c, k0=7.2e-5)
    m = synth.lognormal_area_mult(c.solid)
    p = problem_from_case(c, soc, area_mult=m)
    op = soc.assemble(p)
    ref = soc.steady_state(op)
    with rfb.Solver.from_case(c, area_mult=m) as sv:
        r = sv.solve_nernst(c.s_in, c.eta, 1e-13, max_sweeps=200000)
        s, e = sv.get_state(), sv.get_overpotential()
    assert r["residual"] <= 1e-13
    assert np.abs(s - ref).max() <= 1e-10 * np.abs(ref).max()
    elec = op.unknown & (op.kappa > 0)
    assert np.abs(e[elec] - (op.kin.Vt - np.log(ref[elec] / (1 - ref[elec])))).max() < 1e-7
    assert np.all(e[~elec] == 0.0)
