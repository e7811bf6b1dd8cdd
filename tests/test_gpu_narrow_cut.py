"""Narrow two-sweep tiles cut to each lattice: the same bits as 128-column tiles for the same
cycles, at widths that fall on and beside a cut, heights of one partial and many tiles, batches
whose items are equal shares of all planes and single lattices among them."""
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


@pytest.mark.parametrize("dims", [
    [(24, 20, 37)], [(252, 17, 40)],
    [(16, 70, 25), (20, 16, 24), (36, 36, 37), (68, 45, 41), (80, 83, 33), (92, 92, 50),
     (128, 26, 24), (132, 40, 30), (200, 24, 61)]])
def test_narrow_tiles_are_bitwise_the_128_column_tiles(dims):
    from paper_2502_08034_gb300 import rfb, synth
    cases = [synth.build_case("nc%dx%dx%d" % d, d, 0.82, 4.0, 5 + q, 0.01, -0.10, 0.4, 1e-10,
                              flow_device="cuda") for q, d in enumerate(dims)]
    out = []
    for kernel in (3, 7):
        solvers = [rfb.Solver.from_case(c, area_mult=synth.lognormal_area_mult(c.solid))
                   for c in cases]
        try:
            with rfb.Batch(solvers) as b:
                res, info = b.solve([c.s_in for c in cases], [c.eta for c in cases],
                                    [1e-6] * len(cases), fp32_kernel=kernel, check_every=24)
            assert info["pass_tile_cols"] == (128 if kernel == 3 else 64)
            out.append(([s.get_state() for s in solvers], [r["sweeps"] for r in res]))
        finally:
            for s in solvers:
                s.close()
    assert out[0][1] == out[1][1]
    for x, y in zip(out[0][0], out[1][0]):
        assert np.array_equal(x, y)
