"""The FP64 path's axial form at the sizes and geometries where it can go wrong, against the
oracle: every tail of the 8-half-row and 16-lane tiles (l = 1..7, mixed within a pair), both
outputs, contraction, directions along and against the frames' axes (no azimuth), coincident
centers and P = Q, and batches that mix it with the matrix form.

Bound: 1e-11 of the class's largest integral, the FP64 path's own (each class holds a compact
quartet)."""
import numpy as np
import pytest

import oracle
from paper_2307_03452_gb300 import inputs, lx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


def check(basis, quartets, solid, **kw):
    out, off = lx.eri(basis, quartets, solid=solid, **kw)
    ref, _ = oracle.eri(basis, quartets, solid=solid)
    got = out.cpu().numpy()
    assert np.all(np.isfinite(got))
    l = np.asarray(basis["l"])
    classes = {}
    for i, q in enumerate(np.asarray(quartets)):
        cls = tuple(int(l[s]) for s in q)
        n = int(np.prod([2 * x + 1 if solid else (x + 1) * (x + 2) // 2 for x in cls]))
        classes.setdefault(cls, []).append(np.arange(off[i], off[i] + n))
    for cls, idx in classes.items():
        idx = np.concatenate(idx)
        scale, err = np.abs(ref[idx]).max(), np.abs(got[idx] - ref[idx]).max()
        assert err <= TOL * scale, f"{cls}: {err:.3e} against {scale:.3e}"


@pytest.mark.parametrize("solid", [True, False])
@pytest.mark.parametrize("cls", [(1, 1, 1, 1), (2, 0, 1, 3), (2, 2, 2, 2), (3, 3, 3, 3), (4, 4, 4, 4), (5, 5, 5, 5),
                                 (6, 6, 6, 6), (7, 7, 7, 7), (7, 0, 0, 7), (0, 6, 6, 1), (7, 1, 2, 5), (1, 7, 6, 3)])
def test_classes(cls, solid):
    kmax = 1 if sum(cls) > 20 else 2
    basis, quartets = inputs.uniform_class(cls, 2 if sum(cls) > 20 else 5, 61, cube=1.5, exps=(0.2, 5.0), kmin=1, kmax=kmax)
    check(basis, quartets, solid)


@pytest.mark.parametrize("solid", [True, False])
@pytest.mark.parametrize("cls", [(2, 2, 2, 2), (3, 2, 2, 1), (3, 1, 3, 1), (2, 2, 2, 1), (2, 1, 3, 3), (5, 0, 4, 1)])
def test_contracted_classes_near_the_line(cls, solid):
    # K = 1..5: quartets of one batch on both sides of the line between the two forms, which share pairs
    basis, quartets = inputs.uniform_class(cls, 6, 65, cube=1.5, exps=(0.2, 5.0), kmin=1, kmax=5)
    q = np.asarray(quartets)
    check(basis, np.concatenate([q, np.hstack([q[:, :2], np.roll(q[:, 2:], 1, 0)])]), solid)


@pytest.mark.parametrize("solid", [True, False])
@pytest.mark.parametrize("cls", [(3, 1, 3, 0), (4, 0, 3, 1), (2, 1, 2, 1), (7, 0, 1, 0), (1, 0, 7, 0), (7, 1, 1, 0), (0, 0, 6, 6)])
def test_small_classes_near_the_line(cls, solid):
    # uncontracted classes just above and below the line of either output; (dp|dp) lies below both
    basis, quartets = inputs.uniform_class(cls, 8, 67, cube=1.5, exps=(0.2, 5.0))
    check(basis, quartets, solid)


@pytest.mark.parametrize("solid", [True, False])
def test_directions_without_azimuth(solid):
    # A, B, C, D on the z axis (either order), on the x axis, bra along z and ket along x, tiny
    # tilts of 1e-9 and 1e-170, A = B, C = D, all coincident, P = Q with A != B
    z, x, t = np.array([0, 0, 1.0]), np.array([1.0, 0, 0]), 1e-9
    sets = [[0 * z, z, 2 * z, 3 * z], [3 * z, 2 * z, z, 0 * z], [0 * x, x, 2 * x, 3 * x], [0 * z, z, z + x, z + 2 * x],
            [0 * z, z + t * x, 2 * z, 3 * z - t * x], [0 * z, z + 1e-170 * x, 2 * z, z], [z, z, 0 * z, x], [x, 0 * z, z, z],
            [z, z, z, z], [-z, z, -x, x], [-x, x, -z, z], [0 * z, 1e-170 * x, z, z + 1e-160 * x]]
    n = len(sets)
    ls = np.tile([3, 2, 2, 3], n).astype(np.int32)
    basis = {"l": ls, "nprim": np.ones(4 * n, np.int32), "prim_off": np.arange(4 * n, dtype=np.int32),
             "center": np.concatenate(sets), "exps": np.full(4 * n, 0.7), "coefs": np.ones(4 * n)}
    check(basis, np.arange(4 * n).reshape(n, 4), solid)


def test_mixed_with_the_matrix_form_and_chunked():
    # s and p pairs and K = 16 shells (too many tables) take the matrix form; pairs used by both
    # forms; results do not depend on the workspace
    rng = np.random.default_rng(62)
    ls = np.array([0, 0, 1, 4, 5, 6, 3, 3], np.int32)
    K = np.array([1, 2, 1, 1, 2, 1, 16, 16], np.int32)
    off = np.concatenate([[0], np.cumsum(K)[:-1]]).astype(np.int32)
    basis = {"l": ls, "nprim": K, "prim_off": off, "center": rng.uniform(0, 1.5, (8, 3)),
             "exps": np.exp(rng.uniform(-1.0, 1.5, K.sum())), "coefs": 1 - rng.uniform(0, 1, K.sum())}
    q = [[3, 4, 0, 1], [0, 1, 3, 4], [3, 4, 5, 4], [5, 5, 4, 3], [0, 2, 1, 0], [6, 7, 3, 4], [3, 4, 3, 4], [2, 1, 5, 5]]
    check(basis, q, True)
    b = lx.Batch(basis, q, True)
    outs = []
    for ws in (b.workspace_size(), b.workspace_min(), (b.workspace_size() + b.workspace_min()) // 2):
        outs.append(torch.full((b.out_size,), float("nan"), dtype=torch.float64, device="cuda"))
        b.run(outs[-1], lx.alloc_workspace(ws))
        lx.sync_status()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


def test_far_apart_stays_finite():
    # separations at which F_m, and the powers of the distance, leave the FP64 range
    for d in (1e6, 1e12, 1e160):
        basis, quartets = inputs.uniform_class((6, 5, 6, 7), 1, 63, cube=1.0, exps=(0.5, 2.0))
        basis["center"][2:] += np.array([d, 0.0, 0.0])
        out, _ = lx.eri(basis, quartets, solid=True)
        assert bool(torch.isfinite(out).all()), d


def test_near_and_far_primitives():
    # bra and ket 3 to 14 bohr apart, K = 2 with exponents 0.15 and 6: T of the primitive
    # quartets spans about 1 to 600, so that within one quartet some take the multipole form and
    # some do not (none at 3 bohr, all but one at 14).  Per quartet: 1e-11 of its own largest
    # integral plus 20 times the oracle's noise under a rigid translation, as for far-separated
    # quartets elsewhere.
    seps = [3.0, 5.0, 6.5, 8.0, 10.0, 14.0]
    n = len(seps)
    rng = np.random.default_rng(64)
    ls = np.array([[6, 6, 6, 6], [5, 4, 6, 6], [6, 5, 3, 4], [7, 6, 5, 7], [4, 4, 4, 4], [6, 6, 5, 5]], np.int32).reshape(-1)
    K = np.full(4 * n, 2, np.int32)
    c = rng.uniform(-0.4, 0.4, (n, 4, 3))
    c[:, 2:] += np.array(seps)[:, None, None] * np.array([0.6, 0.0, 0.8])
    basis = {"l": ls, "nprim": K, "prim_off": 2 * np.arange(4 * n, dtype=np.int32), "center": c.reshape(-1, 3),
             "exps": np.tile([0.15, 6.0], 4 * n), "coefs": np.ones(8 * n)}
    quartets = np.arange(4 * n).reshape(n, 4)
    out, off = lx.eri(basis, quartets, solid=True)
    got = out.cpu().numpy()
    ref, _ = oracle.eri(basis, quartets, solid=True)
    ref2, _ = oracle.eri(dict(basis, center=basis["center"] + np.array([0.37, -1.1, 0.53])), quartets, solid=True)
    for i in range(n):
        sl = slice(off[i], off[i] + int(np.prod(2 * ls[4 * i:4 * i + 4] + 1)))
        noise = np.abs(ref[sl] - ref2[sl]).max()
        assert np.abs(got[sl] - ref[sl]).max() <= TOL * np.abs(ref[sl]).max() + 20 * noise, seps[i]


def test_groups_of_one_call_overlap():
    # classes of every group of the main kernel in one call, whose launches overlap: each quartet
    # equals its evaluation alone, bit for bit, in repeated calls and in a replayed graph
    cls = [(7, 7, 7, 7), (6, 6, 6, 6), (5, 5, 5, 5), (4, 4, 4, 4), (3, 3, 3, 3), (4, 3, 7, 7), (7, 6, 2, 1)]
    basis, quartets = inputs.concat([inputs.uniform_class(c, 2, 66 + i, cube=2.0, exps=(0.2, 5.0), kmin=2, kmax=2)
                                     for i, c in enumerate(cls)])
    b = lx.Batch(basis, quartets, True)
    ws = lx.alloc_workspace(b.workspace_size())
    one = torch.cat([lx.eri(basis, [q], solid=True)[0] for q in np.asarray(quartets)])
    out = torch.empty(b.out_size, dtype=torch.float64, device="cuda")
    for _ in range(3):
        out.fill_(float("nan"))
        b.run(out, ws)
        lx.sync_status()
        assert torch.equal(out, one)
    graph = lx.Graph(b, out, ws)
    for _ in range(3):
        out.fill_(float("nan"))
        graph.launch()
        lx.sync_status()
        assert torch.equal(out, one)


@pytest.mark.parametrize("solid", [True, False])
@pytest.mark.parametrize("cls", [(6, 6, 0, 0), (0, 0, 6, 6), (7, 5, 0, 0), (7, 5, 1, 0)])
def test_a_side_of_s_functions(cls, solid):
    # l = 0 alone on one side: tables whose ket blocks are the smallest, several in a row
    basis, quartets = inputs.uniform_class(cls, 5, 68, cube=1.5, exps=(0.2, 5.0), kmin=1, kmax=3)
    check(basis, quartets, solid)
