"""The kernel that timing chooses on lattices beyond the chip (128- or 64-column passes, their
launches overlapping) is bitwise the one-sweep launches, forward and transposed: widths where
64-column tiles are ragged, odd and even sweep counts, many short cycles in a row (each pass
starts while the one before it ends)."""
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


@pytest.mark.parametrize("dims", [(164, 100, 70), (68, 150, 110), (192, 96, 61)])
def test_chosen_pass_is_bitwise_one_sweep_launches(dims):
    from paper_2502_08034_gb300 import rfb, synth
    case = synth.build_case("ap%dx%dx%d" % dims, dims, 0.82, 6.0, 3, 0.01, -0.10, 0.4, 1e-10,
                            flow_device="cuda", flow_tol=1e-10)
    m = synth.lognormal_area_mult(case.solid)
    out, names = [], []
    for kernel in ("plain", "blocked_chunked", "auto"):
        with rfb.Solver.from_case(case, area_mult=m) as sv:
            for n in (2, 4, 7, 2, 2, 60):
                sv.step(case.s_in, case.eta, n, precision="mixed", fp32_kernel=kernel)
            s = sv.get_state()
            # transposed sweeps of the chosen variant (a loose solve first: an adjoint needs one)
            sv.solve(case.s_in, case.eta, 1e-3, precision="fp64", check_every=500)
            dm, _, _ = sv.adjoint("I_tot", 1e-4, precision="mixed", check_every=60)
            out.append((s, dm))
            names.append(sv.tuned_fp32_kernel()[0])
    assert names[2] != "resident"
    for s, dm in out[1:]:
        assert np.array_equal(s, out[0][0])
        assert np.array_equal(dm, out[1][1])
