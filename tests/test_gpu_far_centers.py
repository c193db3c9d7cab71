"""Shell pairs whose centers lie so far apart that their Gaussian prefactor underflows to zero: every
integral is zero, also where powers of the separation leave the FP64 range."""
import numpy as np
import pytest

from paper_2307_03452_gb300 import inputs, lx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("moved", [[1], [2], [0, 2]])
@pytest.mark.parametrize("cls", [(2, 2, 2, 2), (4, 4, 4, 4), (6, 5, 6, 7), (7, 7, 7, 7)])
def test_zero_pairs(cls, moved):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    for d in (1e2, 1e12, 1e24, 1e30, 1e100, 1e160):
        basis, quartets = inputs.uniform_class(cls, 1, 63, cube=1.0, exps=(0.5, 2.0))
        for s in moved:
            basis["center"][s] += np.array([d, 0.0, 0.3 * d])
        out, _ = lx.eri(basis, quartets, solid=True)
        assert bool((out == 0).all()), d
