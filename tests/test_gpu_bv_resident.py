"""The resident Butler-Volmer kernels (a lattice that fits on the chip: one launch per
potential solve, one per cycle of species sweeps) against the oracle at sizes where they can
go wrong: one brick across, ragged bricks, area multipliers; against the launches that larger
lattices take, with a ghost-cell inlet; a cycle longer than one launch; a potential solve cut
off."""
import dataclasses
import functools

import numpy as np
import pytest

from oracle import bv, soc
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
def _case(dims):
    from paper_2502_08034_gb300 import synth
    c = synth.build_case("bvr%dx%dx%d" % dims, dims, 0.82, 4.0, 5, 0.002, -0.10, 0.2, 1e-12,
                         flow_device="cuda")
    return dataclasses.replace(c, k0=2e-5)


@pytest.mark.parametrize("dims", [(5, 6, 9), (13, 11, 15), (21, 8, 10)])
def test_bv_state_matches_the_oracle(dims):
    """Bars of the model's other parity tests: 1e-10 in the concentrations, 1e-7 in phi."""
    from paper_2502_08034_gb300 import rfb, synth
    case = _case(dims)
    m = synth.lognormal_area_mult(case.solid)
    p = problem_from_case(case, soc, area_mult=m)
    C, phi, _ = bv.solve(p, bv.BVParams(), s0=soc.steady_state(soc.assemble(p)), tol=1e-13)
    with rfb.Solver.from_case(case, area_mult=m) as sv:
        sv.solve(case.s_in, case.eta, 1e-13)
        sv.solve_bv(case.s_in, case.eta, 1e-12, start="sbv")
        g = sv.get_bv_state()
    fl = case.solid.ravel() == 0
    for k in ("O", "R", "H"):
        assert np.abs(g[k][fl] - C[k][fl]).max() <= 1e-10 * np.abs(C[k][fl]).max(), k
        assert np.all(g[k][~fl] == 0.0)
    assert np.abs(g["phi"][fl] - phi[fl]).max() <= 1e-7 * np.abs(phi[fl]).max()


def test_resident_and_streamed_kernels_agree():
    """The same solve on a lattice and on the same lattice padded with fluid-free columns
    until nothing fits on the chip: the launches of the larger one are the other path."""
    from paper_2502_08034_gb300 import rfb
    case = _case((13, 11, 15))
    nx, ny, nz = case.dims
    X, Y = 176, 1760                      # 4.6 M cells
    solid = np.ones((nz, Y, X), dtype=np.uint8)
    solid[:, :ny, :nx] = case.solid
    U, V, W = (np.zeros((nz, Y, X + 1)), np.zeros((nz, Y + 1, X)), np.zeros((nz + 1, Y, X)))
    U[:, :ny, :nx], V[:, :ny, :nx], W[:, :ny, :nx] = case.U[:, :, :nx], case.V[:, :ny], case.W
    big = dataclasses.replace(case, dims=(X, Y, nz), solid=solid, U=U, V=V, W=W)
    # beside padding the outer columns of the small lattice are fiber walls: give it those too
    ring = np.ones((nz, ny + 1, nx + 1), dtype=np.uint8)
    ring[:, :ny, :nx] = case.solid
    small = dataclasses.replace(case, dims=(nx + 1, ny + 1, nz), solid=ring,
                                U=U[:, :ny + 1, :nx + 2], V=V[:, :ny + 2, :nx + 1],
                                W=W[:, :ny + 1, :nx + 1])
    out = []
    for c in (small, big):
        with rfb.Solver.from_case(c) as sv:
            sv.solve(c.s_in, c.eta, 1e-9, inlet_bc="ghost")
            r = sv.solve_bv(c.s_in, c.eta, 1e-30, start="sbv", max_sweeps=300, cycle=60,
                            inlet_bc="ghost", allow_not_converged=True)
            g = sv.get_bv_state()
        out.append(([g[k].reshape(c.solid.shape)[:, :ny, :nx] for k in ("O", "R", "H", "phi")], r))
    (a, ra), (b, rb) = out
    # the same iteration in other summation orders, each potential to 1e-13 of its right-hand
    # side: the parity bars
    for x, y, bar in zip(a, b, (1e-10, 1e-10, 1e-10, 1e-7)):
        assert np.abs(x - y).max() <= bar * np.abs(y).max()
    assert ra["I_tot"] == pytest.approx(rb["I_tot"], rel=1e-9)
    assert ra["residual"] == pytest.approx(rb["residual"], rel=1e-6)


def test_cycle_beyond_one_launch_and_a_cut_off_potential_solve():
    from paper_2502_08034_gb300 import rfb
    case = _case((13, 11, 15))
    out = []
    with rfb.Solver.from_case(case) as sv:
        sv.solve(case.s_in, case.eta, 1e-12)
        for cycle in (2500, 2500):        # 2048 sweeps a launch
            r = sv.solve_bv(case.s_in, case.eta, 1e-30, start="sbv", cycle=cycle,
                            max_sweeps=5000, allow_not_converged=True)
            out.append((r["I_tot"], r["phi_min"], r["sweeps"]))
        assert out[0] == out[1] and out[0][2] == 5000
        r = sv.solve_bv(case.s_in, case.eta, 1e-8, start="sbv", max_cg=7, max_sweeps=200,
                        allow_not_converged=True)
        assert r["status"] == rfb.RFB_ERR_NOT_CONVERGED and r["cg_iterations"] == 7 * r["cycles"]
