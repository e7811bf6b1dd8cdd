"""Two-sweep passes with narrow tiles over one lattice, asked for by name, in both launch shapes,
forward and transposed: bitwise the one-sweep launches, on lattices narrower than a tile, with
ragged tiles both ways, one row, many tiles across, odd sweep counts and many short cycles. Every
name that the tuned kernel is reported by can be asked for."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NARROW = ["blocked_narrow_persistent", "blocked_narrow_chunked"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_08034_gb300 import _build
    _build.build()


@functools.lru_cache(maxsize=None)
def _case(dims):
    from paper_2502_08034_gb300 import synth
    return synth.build_case("ns%dx%dx%d" % dims, dims, 0.85, 4.0, 3, 0.01, -0.10, 0.4, 1e-10,
                            flow_device="cuda")


@pytest.mark.parametrize("dims", [(4, 30, 9), (36, 20, 24), (68, 50, 2), (164, 100, 70),
                                  (256, 7, 33), (192, 96, 61)])
def test_narrow_passes_are_bitwise_one_sweep_launches(dims):
    from paper_2502_08034_gb300 import rfb, synth
    case = _case(dims)
    m = synth.lognormal_area_mult(case.solid)
    out = []
    for kernel in ["plain"] + NARROW:
        with rfb.Solver.from_case(case, area_mult=m) as sv:
            for n in (2, 4, 7, 2, 2, 60, 1):
                sv.step(case.s_in, case.eta, n, precision="mixed", fp32_kernel=kernel)
            s = sv.get_state()
            # a loose solve: an adjoint needs one. Transposed sweeps of the kernel named
            sv.solve(case.s_in, case.eta, 1e-3, check_every=500)
            dm, _, r = sv.adjoint("I_tot", 1e-4, precision="mixed", check_every=61,
                                  fp32_kernel="plain" if kernel == "plain" else "auto")
            out.append((s, dm, r["sweeps"]))
            if kernel != "plain":
                assert sv.tuned_fp32_kernel()[0] == kernel
    for s, dm, n in out[1:]:
        assert n == out[0][2] > 0
        assert np.array_equal(s, out[0][0]) and np.array_equal(dm, out[0][1])


@pytest.mark.parametrize("dims", [(36, 20, 24), (33, 18, 41), (164, 100, 70)])
def test_the_reported_kernel_can_be_asked_for(dims):
    from paper_2502_08034_gb300 import rfb
    case = _case(dims)
    with rfb.Solver.from_case(case) as sv:
        sv.step(case.s_in, case.eta, 40, precision="mixed")
        s, name = sv.get_state(), sv.tuned_fp32_kernel()[0]
        sv.reset_state()
        sv.step(case.s_in, case.eta, 40, precision="mixed", fp32_kernel=name)
        assert sv.tuned_fp32_kernel()[0] == name
        assert np.array_equal(sv.get_state(), s)


def test_refusals():
    from paper_2502_08034_gb300 import rfb
    big, odd = _case((164, 100, 70)), _case((33, 18, 41))
    for case, kw in ((big, dict(fp32_kernel="resident")),                # beyond the chip
                     (odd, dict(fp32_kernel=NARROW[0])),                 # nx % 4 != 0
                     (odd, dict(fp32_kernel="resident", dt_mode="global")),
                     (big, dict(fp32_kernel=NARROW[1], dt_mode="global")),
                     (big, dict(fp32_kernel=14))):
        with rfb.Solver.from_case(case) as sv:
            with pytest.raises(rfb.RfbError) as e:
                sv.step(case.s_in, case.eta, 4, precision="mixed", **kw)
            assert e.value.status == rfb.RFB_ERR_INVALID_ARG
