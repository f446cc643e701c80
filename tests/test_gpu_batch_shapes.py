"""GPU checks of the batched solve at the edges of its launch shapes (csrc/batch.cu): 1024,
16384 and 2^20 vectors of four cells in the batch and one size more, and more solves than
blocks' worth of cells.  Each solve against the dense solver's: both within 1e-8 ||f|| of the
solution, 1e3 for the operator's inverse."""
import pytest
import torch

from paper_1305_2418_gb300 import build, mgfr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU test run without a GPU"
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("sizes", [[8], [16, 16], [16, 8, 16], [32] * 4, [32] * 4 + [8],
                                   [128] * 4, [8] + [128] * 4, [8] * 30],
                         ids=lambda v: f"{len(v)}x{max(v)}")
def test_shapes(dev, sizes):
    ds = [torch.from_numpy(synth.lognormal_delta(N, 3.0 * N, 1.5, 700 + q)).to(dev)
          for q, N in enumerate(sizes)]
    boxes = [3.0 * N for N in sizes]
    s = mgfr.Solver(0, precision=mgfr.PREC_MIXED)
    outs, st = s.batch_solve(ds, boxes, [1e-5] * len(sizes))
    assert st == mgfr.MGFR_OK
    one = mgfr.Solver(0, fr0_abs=1e-5)
    for d, box, o in zip(ds, boxes, outs):
        assert o["stats"]["res_l2_final"] <= 1e-8 * o["stats"]["f_l2"]
        assert float((o["fr"] / one.solve_density(d, box)["fr"] - 1.0).abs().max()) <= 1e-5
    one.close()
    s.close()
