"""Temperature solve (rt_newton.cuh) against the oracle's Newton: lane segments and their edges, channels
of weight zero, hot and cold right-hand sides (FP32 root with one Halley step, FP64 polish and fallback).

Both solve to |dT| <= 1e-14 T in FP64; the balance's own conditioning leaves a few units of 1e-15 times
the cancellation in its sums, so 1e-12 holds everywhere.
"""
import dataclasses

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [1, 2, 3, 4, 7, 8, 16, 17, 33, 64, 65, 130])
@pytest.mark.parametrize("level", [1.0, 1e-12, 1e9, 1e-40])
def test_temperature_matches_oracle(F, level):
    import torch

    import paper_2306_05789_gb300 as rt
    from oracle import oracle as O
    fr = W.midpoint_freqs(F, albedo=0.3, c_offset=None)
    if F > 2:
        fr.albedo[1] = 1.0   # a channel that has no say
    p = W.cube_problem(3, W.Kappa(W.KAPPA_CONST, 0.0, 0.0), fr, R0=0.0, T_emit=1.0)
    p = dataclasses.replace(p, Q0=level)
    # kappa = 0: J is the source after one step, T its balance
    op = rt.rt_build_operator(p, rt.hparams(mode=rt.RT_MODE_DENSE, prec=rt.RT_PREC_F64))
    J = torch.zeros(F, p.N, dtype=torch.float64, device="cuda")
    T = torch.zeros(p.N, dtype=torch.float64, device="cuda")
    op.solve_fixed_point(J, T, tol=1e-10, max_iter=8)
    ref = O.temperature_newton(J.cpu().numpy(), fr)
    got = T.cpu().numpy()
    assert np.all(np.abs(got - ref) <= 1e-12 * np.maximum(ref, 1e-300))
    op.free()
