"""Row and column evaluation (rt_rows.cuh): every evaluator and chunk width against the oracle.

With eta tiny every leaf pair is a dense block, so an apply shows the row evaluation alone: pass and
sub-cluster edges (tetrahedra per pass 128 or 512, leaves up to 256 columns), group chunks (1, 4, 8,
16, several) and the three evaluators (phase tables: walls normal to an axis; plain: oblique walls, a
wall that makes the domain's box too long, node sums; general: two walls, grid).  With eta = 2 the
pivot columns take part.

Tolerances.  FP32 entries carry about ten roundings of 6e-8 and an optical depth within 1e-6 of its
value (the bound of the special-function sines), so an apply to positive vectors is within 2e-6 of the
dense FP64 matrix in the 2-norm; ACA at eps = 1e-4 adds its own 1e-4 bound.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _problem(n, groups, wall, kind="sin"):
    rng = np.random.default_rng(n + 10 * groups)
    kappa = W.sinprod_kappa(0.6) if kind != "const" else W.Kappa(W.KAPPA_CONST, 1.3, 0.0)
    p = W.cube_problem(n, kappa, W.midpoint_freqs(groups, albedo=0.3), R0=0.0)
    xyz = p.xyz.copy()
    inner = ((xyz > 1e-9) & (xyz < 1 - 1e-9)).all(axis=1)
    xyz[inner] += rng.uniform(-0.1, 0.1, size=(int(inner.sum()), 3)) / (n - 1)
    p.xyz = xyz
    if wall:
        p.wall = W.Wall(*wall)
    if kind == "uneven":
        p.freqs.c = np.linspace(0.5, 1.0, groups) ** 2 + 0.3
    if kind == "grid":
        p.kappa = W.Kappa(W.KAPPA_GRID, 0.0, 0.0, rng.uniform(0.2, 2.0, size=(3, 4, 5)).astype(np.float32),
                          (0.0, 0.0, 0.0, 1.0, 1.0, 1.0))
        p.more_walls = (W.Wall((0.0, 0.0, 0.0), (0.0, -1.0, 0.0), 0.4),)
        p.corner = True
    return p


Z0 = ((0.0, 0.0, 0.0), (0.0, 0.0, -1.0), 0.5)
X1 = ((1.0, 0.3, 0.0), (2.0, 0.0, 0.0), 0.7)
Y_OFF = ((0.0, -0.015, 0.0), (0.0, -1.0, 0.0), 0.6)
OBLIQUE = ((0.0, 0.0, 0.0), (-0.3, -0.2, -1.0), 0.5)


@pytest.mark.parametrize("n,groups,wall,kind,leaf", [
    (2, 1, Z0, "sin", 64), (5, 1, None, "sin", 64), (8, 1, Z0, "sin", 256), (7, 1, X1, "const", 33),
    (6, 2, X1, "sin", 64), (7, 4, Y_OFF, "sin", 31), (7, 5, Z0, "sin", 64), (6, 9, Z0, "uneven", 64),
    (8, 16, Z0, "sin", 100), (6, 17, X1, "sin", 64), (5, 33, Z0, "sin", 64),
    (6, 1, OBLIQUE, "sin", 64), (6, 8, OBLIQUE, "sin", 64), (6, 20, OBLIQUE, "sin", 64),
    (6, 1, Z0, "grid", 64), (6, 6, Z0, "grid", 64), (5, 18, Z0, "grid", 64),
])
@pytest.mark.parametrize("eta", [1e-9, 2.0])
def test_rows_and_columns_match_oracle(n, groups, wall, kind, leaf, eta):
    import torch

    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    p = _problem(n, groups, wall, kind)
    X = W.rand_vectors((groups, p.N), seed=1).astype(np.float32)
    ref = O.DenseOperator(p).apply(X.astype(np.float64))
    op = rt.rt_build_operator(p, rt.hparams(leaf=leaf, eta=eta))
    Xd = torch.tensor(X, device="cuda")
    Y = torch.empty_like(Xd)
    op.apply(Xd, Y)
    err = np.linalg.norm(Y.double().cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err < (2e-6 if eta < 1 else 1e-4)
    op.free()


@pytest.mark.parametrize("groups", [1, 6])
def test_aca_resumes_when_the_term_pool_runs_out(groups):
    """eps = 1e-6 needs more terms than the pool first holds (24 a block): blocks stop, the pool grows,
    they go on (one group: ranks above 24).  With six groups every block here ends dense."""
    import torch

    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    p = _problem(11, groups, Z0)
    X = W.rand_vectors((groups, p.N), seed=1).astype(np.float32)
    rows = np.arange(0, p.N, 7, dtype=np.int32)
    c, g = np.unique(np.asarray(p.freqs.c), return_inverse=True)
    ref = np.stack([np.einsum("ij,j->i", np.asarray(O.G_rows(p, rows, c=c))[:, g[f]], X[f].astype(np.float64))
                    for f in range(groups)])
    for wave_bytes in (0, 1 << 20):
        op = rt.rt_build_operator(p, rt.hparams(leaf=40, aca_eps=1e-6, wave_bytes=wave_bytes))
        Xd = torch.tensor(X, device="cuda")
        Y = torch.empty_like(Xd)
        op.apply(Xd, Y)
        got = Y.double().cpu().numpy()[:, rows]
        assert np.linalg.norm(got - ref) < 4e-6 * np.linalg.norm(ref)
        op.free()


def _apply(op, X):
    import torch
    Xd = torch.tensor(X, device="cuda")
    Y = torch.empty_like(Xd)
    op.apply(Xd, Y)
    return Y.double().cpu().numpy()


@pytest.mark.parametrize("groups", [1, 3, 17])
@pytest.mark.parametrize("one_block_waves", [False, True])
def test_aca_of_high_rank_grows_the_pool_many_times(groups, one_block_waves):
    """Touching blocks of 166 to 666 rows at a tolerance below FP32: every block runs to the rank where
    dense storage is smaller (83 to 332 terms), so the pool, 24 terms a block at first, grows six times
    in one wave and four to seven with one block to a wave; the terms' 16-byte accesses need every
    capacity rounded.  All blocks end dense, and the apply is that of the dense matrix."""
    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    p = _problem(11, groups, Z0)
    X = W.rand_vectors((groups, p.N), seed=1).astype(np.float32)
    rows = np.arange(0, p.N, 7, dtype=np.int32)
    c, g = np.unique(np.asarray(p.freqs.c), return_inverse=True)
    ref = np.stack([np.einsum("ij,j->i", np.asarray(O.G_rows(p, rows, c=c))[:, g[f]], X[f].astype(np.float64))
                    for f in range(groups)])
    _, blocks, _ = rt.rt_plan(p.xyz, 200, 2.0, rt.RT_ADM_CENTER)
    far = blocks[blocks[:, 4] == 1].astype(np.int64)
    op = rt.rt_build_operator(p, rt.hparams(leaf=200, adm=rt.RT_ADM_CENTER, aca_eps=1e-9,
                                            wave_bytes=1 if one_block_waves else 0))
    info = op.info()
    got = _apply(op, X)[:, rows]
    op.free()
    assert info["aca_waves"] == (len(far) if one_block_waves else 1)
    assert info["n_far"] == 0 and info["n_dense_fallback"] == len(far)
    # (m + n) floats a term and group: what the blocks took, beyond the capacity after five growths by half
    assert info["entries_evaluated"] - p.N ** 2 > 24 * 1.5 ** 5 * (far[:, 1] + far[:, 3]).sum()
    assert np.linalg.norm(got - ref) < 2e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("scale,wall", [(1.0, X1), (0.6, ((0.6, 0.3, 0.0), (1.0, 0.0, 0.0), 0.7)), (1.0, Z0)])
def test_tetrahedron_flat_against_a_wall(scale, wall):
    """A boundary sliver 1e-9 high lies in the wall's plane once rounded to FP32: rows of vertices on the
    wall have a reflected path of zero height to it, which must not reach the sums as NaN."""
    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    p = _problem(6, 1, wall)
    p.xyz = p.xyz * scale
    axis = int(np.argmax(np.abs(wall[1])))
    at = wall[0][axis]
    face = np.flatnonzero(np.abs(p.xyz[:, axis] - at) < 1e-12)
    u, v = [d for d in range(3) if d != axis]
    corner = face[np.argsort(p.xyz[face, u] + p.xyz[face, v])[:3]]   # three vertices at one corner of the face
    tip = np.array([0.5, 0.3, 0.2]) @ p.xyz[corner]   # on no quadrature point of the sliver
    tip[axis] = at + (1e-9 if at == 0.0 else -1e-9)
    p.tet = np.vstack([p.tet, [[*corner, p.N]]]).astype(np.int32)
    p.xyz = np.vstack([p.xyz, tip])
    X = W.rand_vectors((1, p.N), seed=1).astype(np.float32)
    ref = O.DenseOperator(p).apply(X.astype(np.float64))
    op = rt.rt_build_operator(p, rt.hparams(eta=1e-9))
    got = _apply(op, X)
    op.free()
    assert np.isfinite(got).all()
    assert np.linalg.norm(got - ref) < 2e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("groups", [1, 3])
def test_blocks_of_several_groups_resume_and_stay_compressed(groups):
    """eps = 1e-6 takes more than 24 terms a block on average here, so the pool grows, blocks of several
    groups go on in the larger one, and all of them end compressed.  Tolerance: eps for the far field
    plus 2e-6 for FP32 entries."""
    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    p = _problem(14, groups, Z0)
    X = W.rand_vectors((groups, p.N), seed=1).astype(np.float32)
    rows = np.arange(0, p.N, 11, dtype=np.int32)
    c, g = np.unique(np.asarray(p.freqs.c), return_inverse=True)
    ref = np.stack([np.einsum("ij,j->i", np.asarray(O.G_rows(p, rows, c=c))[:, g[f]], X[f].astype(np.float64))
                    for f in range(groups)])
    _, blocks, _ = rt.rt_plan(p.xyz, 180, 2.0)
    far, near = (blocks[blocks[:, 4] == k].astype(np.int64) for k in (1, 0))
    op = rt.rt_build_operator(p, rt.hparams(leaf=180, aca_eps=1e-6))
    info = op.info()
    got = _apply(op, X)[:, rows]
    op.free()
    assert info["n_far"] == len(far) > 0 and info["n_dense_fallback"] == 0
    used = info["entries_evaluated"] - (near[:, 1] * near[:, 3]).sum()
    assert used > 24 * (far[:, 1] + far[:, 3]).sum()
    assert np.linalg.norm(got - ref) < 3e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("k0,c", [(50.0, (3.0, 2.0, 1.0)), (12.0, tuple(range(8, 0, -1))), (12.0, tuple(range(1, 9))),
                                  (12.0, tuple(np.linspace(4.0, 0.25, 16)))])
@pytest.mark.parametrize("wall", [Z0, OBLIQUE])
def test_equally_spaced_scales_in_either_order_at_large_depth(k0, c, wall):
    """Equally spaced group scales, ascending and descending, with optical depths up to 90 per unit scale:
    every group is finite and agrees with the oracle between opposite faces too, where exp(-c tau) of the
    larger scales is far below the FP32 range.

    Tolerance: an FP32 optical depth is within 1e-6 of its value in relative terms, so a value
    exp(-c tau) above 1e-30 (c tau < 70) is within 7e-5."""
    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    p = _problem(6, len(c), wall, kind="const")
    p.kappa.k0 = k0
    p.freqs.c = np.array(c, dtype=np.float64)
    ref_op = O.DenseOperator(p)
    X = W.rand_vectors((len(c), p.N), seed=1).astype(np.float32) + np.float32(0.5)
    far = X * (p.xyz[:, 0] > 0.79)
    rows = p.xyz[:, 0] < 0.21
    for eta in (1e-9, 2.0):
        op = rt.rt_build_operator(p, rt.hparams(eta=eta))
        for V, on in ((X, np.ones(p.N, dtype=bool)), (far, rows)):
            ref = ref_op.apply(V.astype(np.float64))[:, on]
            got = _apply(op, V)[:, on]
            assert np.isfinite(got).all()
            if eta > 1:
                continue
            for g in range(len(c)):
                size = np.linalg.norm(ref[g])
                assert np.linalg.norm(got[g] - ref[g]) <= 7e-5 * size + 1e-30 * p.N, (g, size)
        op.free()


@pytest.mark.parametrize("wall,kind", [(Z0, "sin"), (Z0, "const"), (OBLIQUE, "sin"), (Z0, "grid")])
def test_entries_are_not_shifted_by_the_rounding_of_a_group_scale(wall, kind):
    """Scales just below and just above the middle between two FP32 numbers round 5.8e-8 apart from their
    values in opposite directions.  The mean relative error over all entries, in which every other
    rounding is the same up to 1/sqrt(entries), may differ by 2e-8 between the two."""
    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    mean = []
    for c in (1.0 + 0.49 * 2.0 ** -23, 1.0 + 0.51 * 2.0 ** -23):
        p = _problem(7, 1, wall, kind)
        p.freqs.c = np.array([c])
        ref = O.DenseOperator(p)
        op = rt.rt_build_operator(p, rt.hparams(eta=1e-9))
        err = 0.0
        for j in range(p.N):
            x = np.zeros((1, p.N), dtype=np.float32)
            x[0, j] = 1.0
            col = ref.G[0][:, j]
            rel = (_apply(op, x)[0] - col) / col
            err += float(np.median(rel)) / p.N   # a column's middle: the grid's kinks have a long tail
        mean.append(err)
        op.free()
    assert abs(mean[0] - mean[1]) < 2e-8, mean


@pytest.mark.parametrize("groups", [1, 4, 5, 8, 9, 17])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("kind", ["const", "sin", "grid"])
def test_dense_matrix_of_every_group_chunk_matches_oracle(groups, prec, kind):
    """Dense mode at the edges of its instances (1, 4, 8 and 16 groups a pass).  FP64: sums of positive
    terms with about ten roundings each and a depth within 1e-14; FP32 as the rows above."""
    import torch

    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    f64 = prec == "f64"
    p = _problem(5, groups, Z0, kind)
    X = W.rand_vectors((groups, p.N), seed=1)
    X = X if f64 else X.astype(np.float32)
    ref = O.DenseOperator(p).apply(X.astype(np.float64))
    op = rt.rt_build_operator(p, rt.hparams(mode=rt.RT_MODE_DENSE, prec=rt.RT_PREC_F64 if f64 else rt.RT_PREC_F32))
    got = _apply(op, X)
    op.free()
    assert np.linalg.norm(got - ref) < (1e-13 if f64 else 2e-6) * np.linalg.norm(ref)


def test_dense_sums_that_overflow_are_infinite():
    """Cells of 2e13 units a side have volumes beyond FP32: the FP32 dense matrix is infinite throughout,
    not NaN (positive terms only)."""
    import paper_2306_05789_gb300 as rt
    p = _problem(4, 2, Z0, "const")
    p.xyz = p.xyz * 6e13
    p.kappa.k0 = 1e-14
    op = rt.rt_build_operator(p, rt.hparams(mode=rt.RT_MODE_DENSE, prec=rt.RT_PREC_F32))
    got = _apply(op, np.ones((2, p.N), dtype=np.float32))
    op.free()
    assert np.isposinf(got).all()
