"""Split-precision panels whose results lie near the ends of the exponent range
(the epilogue's general form) beside ordinary rows and zero rows, with columns
of U that cancel (small sums, converted without dropping bits) or vanish:
bitwise against the emulation of the digit scheme."""
import numpy as np
import pytest

from tests.test_gpu_panel import emulate, make_case, to_panel, to_u

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,w,layout", [(150, 128, "col"), (130, 100, "row"), (40, 64, "col"), (33, 20, "row")])
@pytest.mark.parametrize("every", [1, 40])
def test_exponent_range(rows, w, layout, every):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as gbr
    Y, U = make_case(rows, w, seed=rows + w + every)
    Y[::every] *= (2.0 ** np.array([-900, -700, 0, 700, 900]))[np.arange(len(Y[::every])) % 5][:, None]
    Y[3] = 0.0
    U[:, 5] = 0.0
    U[:, 6] = 0.0
    U[0, 6], U[1, 6] = 1.0, -1.0
    Y[:, 1] = Y[:, 0] * (1.0 + 2.0 ** -40)  # column 6 cancels 40 bits
    t = to_panel(Y, layout)
    gbr.update_panel(t, to_u(U), "ozaki")
    got, want = t.cpu().numpy(), emulate(Y, U)
    assert np.array_equal(got.view(np.uint64), want.view(np.uint64))
