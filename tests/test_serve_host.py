"""Host-side checks of the serving entry points (no GPU needed): option
validation, rejection of a request whose estimated footprint exceeds the
budget, and unknown request ids."""
from __future__ import annotations

import pytest

import paper_2306_05789_gb300 as rt
import workloads as W


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2306_05789_gb300 import build
    build.build()


def test_invalid_server_options_are_rejected():
    for kw in ({"hbm_budget": 0}, {"slots": 0}, {"slots": 65}, {"max_bypass": -1}, {"tol": -1.0}):
        with pytest.raises(rt.RtError) as e:
            rt.Server(rt.hparams(), **kw)
        assert e.value.code == rt.RT_EINVAL
    with pytest.raises(rt.RtError):
        rt.Server(rt.hparams(mode=rt.RT_MODE_DENSE, prec=rt.RT_PREC_F64))


def test_request_larger_than_the_budget_is_refused_at_submit():
    srv = rt.Server(rt.hparams(), hbm_budget=1000, slots=1)
    p = W.cube_problem(8, W.sinprod_kappa(0.5), W.midpoint_freqs(2), R0=0.5)
    with pytest.raises(rt.RtError) as e:
        srv.submit(p)
    assert e.value.code == rt.RT_ENOMEM
    assert srv.info()["submitted"] == 0
    srv.free()


def test_malformed_request_and_unknown_id_are_rejected():
    srv = rt.Server(rt.hparams(), hbm_budget=10**9, slots=1)
    p = W.cube_problem(6, W.sinprod_kappa(0.5), W.midpoint_freqs(1), R0=0.5)
    p.tet[0, 0] = p.N + 5
    with pytest.raises(rt.RtError) as e:
        srv.submit(p)
    assert e.value.code == rt.RT_EINVAL
    srv._dims[12345] = (1, 8)
    with pytest.raises(rt.RtError) as e:
        srv.poll(12345)
    assert e.value.code == rt.RT_EINVAL
    srv.free()


def _estimate(p, hp):
    srv = rt.Server(hp, hbm_budget=1, slots=1)
    with pytest.raises(rt.RtError) as e:
        srv.submit(p)
    srv.free()
    assert e.value.code == rt.RT_ENOMEM
    return int(str(e.value).split("estimated ")[1].split()[0])


@pytest.mark.parametrize("n,F", [(6, 1), (12, 1), (10, 5)])
def test_the_estimate_covers_the_tables_beside_the_near_blocks(n, F):
    """No admissible block: while the near blocks are filled, the device holds them, the mesh (116 bytes
    a tetrahedron, 60 a vertex), the evaluation tables (144 bytes a tetrahedron, 32 a vertex, and 12
    for every tetrahedron of every sub-cluster, at least one each)."""
    p = W.cube_problem(n, W.sinprod_kappa(0.5), W.midpoint_freqs(F), R0=0.5)
    N, T = p.N, p.tet.shape[0]
    held = 4 * F * N * N + 116 * T + 60 * N + 144 * T + 32 * N + 12 * T
    est = _estimate(p, rt.hparams(eta=1e-9))
    assert held <= est <= 1.5 * held + (1 << 20)
    # further walls take smaller tables
    p.more_walls = (W.wall_y0(0.4),)
    assert held - 96 * T <= _estimate(p, rt.hparams(eta=1e-9)) <= est


def test_the_estimate_covers_a_growing_term_pool():
    """At eps = 1e-8 blocks take 48 terms: pools of 24, 36 and 54 terms a block, two of them at once."""
    p = W.cube_problem(16, W.sinprod_kappa(0.5), W.midpoint_freqs(2), R0=0.5)
    _, blocks, _ = rt.rt_plan(p.xyz, 64, 2.0)
    far = blocks[blocks[:, 4] == 1].astype("int64")
    term = 2 * 4 * (far[:, 1] + far[:, 3]).sum()
    fine, coarse = (_estimate(p, rt.hparams(aca_eps=e)) for e in (1e-8, 1e-4))
    assert fine >= (36 + 54 + 48) * term
    assert coarse >= (24 + 24) * term
