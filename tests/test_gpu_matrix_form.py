"""Quartets of the FP64 path that take the matrix form: small classes, and deep contractions whose
tables would not fit the axial form's room.  Every GEMM tile shape against the oracle and against each other
(odd and large row and column counts), J and K straight from [ab|q] (jk_direct_kernel), and lists that
hold both forms, whose pairs and workspace they share.

Launch counts say which form ran: a list in the matrix form alone launches one GEMM2 per tile shape and
one pair kernel; the axial form launches two rotations there, and a list with both forms two pair kernels.

Bounds: integrals 1e-11 of their class's largest (the FP64 path's own), J and K as in test_gpu_jk."""
import numpy as np
import pytest

import oracle
from paper_2307_03452_gb300 import inputs, lx

from test_gpu_jk import density, weights

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)
    lx.tune_clear()
    yield
    lx.tune_clear()


def make(specs, seed, cube=1.5):
    """One quartet per (l, K) specification (four of each)."""
    rng = np.random.default_rng(seed)
    parts = []
    for ls, ks in specs:
        K = np.asarray(ks, np.int32)
        off = np.concatenate([[0], np.cumsum(K)[:-1]]).astype(np.int32)
        basis = {"l": np.asarray(ls, np.int32), "nprim": K, "prim_off": off, "center": rng.uniform(0, cube, (4, 3)),
                 "exps": np.exp(rng.uniform(np.log(0.2), np.log(5.0), K.sum())), "coefs": 1 - rng.uniform(0, 1, K.sum())}
        parts.append((basis, np.arange(4, dtype=np.int32)[None]))
    return inputs.concat(parts)


def run(batch):
    out = torch.full((batch.out_size,), float("nan"), dtype=torch.float64, device="cuda")
    lx.stage_times()
    batch.run(out, lx.alloc_workspace(batch.workspace_size()), time_stages=True)
    lx.sync_status()
    return out, lx.stage_times()[1]


# rows from 1 to 135 and 168, columns from 1 to 143 and 210: one and several tiles of each shape, edges of one row or
# column (N = 1 mod 8) and of more
SOLID = [((7, 4, 0, 0), (1, 1, 8, 8)), ((6, 5, 0, 0), (1, 1, 16, 5)), ((0, 0, 6, 5), (8, 8, 1, 1)),
         ((3, 2, 3, 2), (16, 6, 8, 5)), ((2, 2, 2, 2), (8, 8, 8, 8)), ((2, 1, 2, 1), (2, 1, 1, 3)), ((1, 1, 1, 1), (1, 1, 1, 1)),
         ((0, 0, 0, 0), (3, 2, 1, 1)), ((2, 0, 1, 0), (1, 2, 2, 1))]
CART = [((6, 2, 0, 0), (1, 1, 1, 1)), ((4, 3, 0, 0), (1, 1, 2, 1)), ((0, 0, 5, 3), (1, 1, 1, 1)), ((0, 0, 4, 4), (1, 1, 1, 1)),
        ((2, 2, 2, 2), (8, 8, 8, 4)), ((2, 1, 2, 1), (2, 1, 1, 1)), ((1, 1, 1, 1), (1, 1, 1, 1)), ((0, 0, 0, 0), (3, 2, 1, 1))]


@pytest.mark.parametrize("solid", [True, False])
def test_every_tile_shape(solid):
    specs = SOLID if solid else CART
    basis, quartets = make(specs, 71)
    b = lx.Batch(basis, quartets, solid)
    ref, off = oracle.eri(basis, quartets, solid=solid)
    first = None
    for v1 in range(4):
        v2 = 3 - v1
        lx.tune_import([tuple(l) + (k[0] * k[1], k[2] * k[3], int(solid), v1, v2) for l, k in specs])
        out, launches = run(b)
        assert launches["pair_h"] == 1 and launches["gemm1"] == 1 and launches["gemm2"] == 1  # the matrix form alone
        got = out.cpu().numpy()
        for i, (l, k) in enumerate(specs):
            sl = slice(off[i], off[i] + int(b.sizes[i]))
            assert np.abs(got[sl] - ref[sl]).max() <= TOL * np.abs(ref[sl]).max(), (l, k, v1, v2)
        first = out if first is None else first
        assert torch.equal(out, first), (v1, v2)
    lx.tune_clear()


def check_jk(basis, q, solid, sym, limit=None):
    """J and K against the oracle's; returns the launch counts."""
    _, nbf = oracle.function_offsets(basis, solid)
    D = density(nbf, 73, sym=sym)
    Jr, Kr = oracle.jk(basis, q, D, solid)
    jb = lx.JKBatch(basis, q, solid)
    J, K = (torch.zeros(nbf, nbf, dtype=torch.float64, device="cuda") for _ in range(2))
    lx.stage_times()
    jb.run_jk(torch.tensor(D, device="cuda"), J, K, lx.alloc_workspace(limit or jb.workspace_size()), time_stages=True)
    lx.sync_status()
    launches = lx.stage_times()[1]
    WJ, WK = weights(basis, q, D, solid)
    ref, _ = oracle.eri(basis, q, solid=solid)
    ints, _ = lx.eri(basis, q, solid=solid)
    per_int = np.abs(ints.cpu().numpy() - ref).max()
    assert per_int <= TOL * np.abs(ref).max()
    tol = per_int + 1e-14 * np.abs(ref).max()
    assert np.all(np.abs(J.cpu().numpy() - Jr) <= tol * WJ)
    assert np.all(np.abs(K.cpu().numpy() - Kr) <= tol * WK)
    assert np.abs(Jr).max() > 0 and np.abs(Kr).max() > 0
    return launches


def small_basis(ls, seed, kmax=3):
    rng = np.random.default_rng(seed)
    K = rng.integers(1, kmax + 1, len(ls)).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(K)[:-1]]).astype(np.int32)
    return {"l": np.asarray(ls, np.int32), "nprim": K, "prim_off": off, "center": rng.uniform(0, 2.0, (len(ls), 3)),
            "exps": np.exp(rng.uniform(np.log(0.2), np.log(5.0), K.sum())), "coefs": 1 - rng.uniform(0, 1, K.sum())}


@pytest.mark.parametrize("solid", [True, False])
def test_jk_of_small_classes(solid):
    # s, p and d shells, one d at most on each side: every class lies below the lines
    basis = small_basis([0, 1, 2, 1, 0, 2], 74)
    rng = np.random.default_rng(75)
    pairs = [(0, 1), (1, 3), (2, 0), (1, 2), (4, 4), (5, 3), (0, 5), (3, 3)]
    q = np.array([pairs[i] + pairs[j] for i, j in rng.integers(0, len(pairs), (24, 2))] + [(0, 0, 0, 0), (2, 1, 2, 1)],
                 np.int32)
    launches = check_jk(basis, q, solid, sym=not solid)
    assert launches["pair_h"] == 1 and launches["gemm2"] == 0 and launches["digest"] == 1


@pytest.mark.parametrize("solid", [True, False])
def test_jk_of_deep_contractions(solid):
    # 2,048 and 4,096 primitive quartets of (dd|dd), above the line, in the matrix form for their tables' size
    basis, quartets = make([((2, 2, 2, 2), (8, 8, 8, 8) if solid else (8, 8, 8, 4))], 76)
    launches = check_jk(basis, np.asarray(quartets), solid, sym=solid)
    assert launches["pair_h"] == 1 and launches["gemm2"] == 0 and launches["digest"] == 1


@pytest.mark.parametrize("solid", [True, False])
def test_jk_of_both_forms(solid):
    # g, f and d shells among s and p ones: one list in both forms, digested by both kernels, in one chunk and
    # one quartet at a time
    basis = small_basis([4, 0, 3, 1, 2, 4], 77, kmax=2)
    rng = np.random.default_rng(78)
    q = rng.integers(0, 6, (20, 4)).astype(np.int32)
    q[0], q[1], q[2], q[3] = [0, 5, 0, 5], [1, 3, 1, 1], [0, 5, 1, 3], [1, 3, 0, 5]
    launches = check_jk(basis, q, solid, sym=not solid)
    assert launches["pair_h"] == 2 and launches["digest"] == 2
    check_jk(basis, q, solid, sym=not solid, limit=lx.JKBatch(basis, q, solid).workspace_min())
