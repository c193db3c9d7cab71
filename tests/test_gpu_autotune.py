"""Autotuning of batches that hold both forms of the FP64 path: the tuning table is for quartets that
take the GEMMs, so their keys are the ones timed and recorded, however cheap beside the others."""
import numpy as np
import pytest

from paper_2307_03452_gb300 import inputs, lx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)
    lx.tune_clear()
    yield
    lx.tune_clear()


@pytest.mark.parametrize("solid", [True, False])
@pytest.mark.parametrize("max_keys", [1, 4])
def test_only_keys_of_the_gemms_are_recorded(solid, max_keys):
    # (pp|pp) and (ds|pp) lie far below the lines of the axial form, (hh|hh) and (ii|gg) far above
    parts = [inputs.uniform_class(c, 3, 90 + i, cube=2.0, exps=(0.2, 5.0))
             for i, c in enumerate([(5, 5, 5, 5), (1, 1, 1, 1), (6, 6, 4, 4), (2, 0, 1, 1)])]
    basis, quartets = inputs.concat(parts)
    b = lx.Batch(basis, quartets, solid)
    out = torch.empty(b.out_size, dtype=torch.float64, device="cuda")
    ws = lx.alloc_workspace(b.workspace_size())
    b.run(out, ws)
    lx.sync_status()
    ref = out.clone()
    rows = lx.autotune(b, max_keys=max_keys, samples=3)
    got = {tuple(int(x) for x in r[:4]) for r in np.asarray(rows)}
    want = {(1, 1, 1, 1), (2, 0, 1, 1)}
    assert got <= want and len(got) == min(max_keys, 2)
    out.fill_(float("nan"))
    b.run(out, ws)
    lx.sync_status()
    assert torch.equal(out, ref)
