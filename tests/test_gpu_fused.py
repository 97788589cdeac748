"""Fused acoustic kernels (acoustic_fused.cu) against the FP64 oracle where
they can go wrong: grids that end on, just before and just past a tile or a
4-cell group, borders narrower than the stencil's reach, step counts that
leave a short last launch, receivers on every part of the interior, and shot
counts that select each launch variant.  Tolerances are the suite's own for
seismograms and adjoint sources (1e-4 relative L2) and gradients (1e-3).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_14189_gb300 import inputs

pytestmark = pytest.mark.gpu

# (nz, nx, pml, nt, shots): padded widths 72 = 3 x 24, 64 = 2 x 32, 73, 71,
# 45; borders 0, 2, 3; 101 and 40 steps (2 and 3 steps a launch); on the small
# grids 1 to 150 shots run from one CTA per SM to two waves of three
CASES = [
    (52, 52, 10, 101, 1), (44, 44, 10, 100, 2), (30, 53, 10, 101, 2), (61, 51, 10, 61, 1),
    (33, 39, 3, 101, 2), (41, 52, 2, 100, 1), (40, 45, 0, 61, 2), (9, 11, 20, 100, 1),
    (17, 19, 6, 40, 40), (17, 19, 6, 40, 80), (17, 19, 6, 41, 150),
]


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def setup(nz, nx, pml, nt, shots):
    rng = np.random.default_rng(nz * 1000 + nx)
    v = np.clip(2200 + 300 * rng.standard_normal((nz, nx)), 1500, 3300).astype(np.float32)
    src = np.stack([rng.integers(0, nz, shots), rng.integers(0, nx, shots)], -1).astype(np.int32)
    rec = np.stack([rng.integers(0, nz, (shots, 24)), rng.integers(0, nx, (shots, 24))],
                   -1).astype(np.int32)
    rec[:, 0], rec[:, 1] = (0, nx - 1), (nz - 1, 0)
    rec[:, 3] = rec[:, 2]  # two receivers on one cell
    w = np.stack([inputs.ricker(25.0, 1e-3, nt)] * shots).astype(np.float32)
    d_obs = (0.01 * rng.standard_normal((shots, 24, nt))).astype(np.float32)
    return v, w, src, rec, d_obs


@pytest.mark.parametrize("case", CASES, ids=str)
def test_fused_matches_oracle(case):
    from paper_2604_14189_gb300 import sweep
    nz, nx, pml, nt, shots = case
    v, w, src, rec, d_obs = setup(*case)
    p = sweep.problem(nz=nz, nx=nx, pml=pml, dx=10.0, dt=1e-3, nt=nt, nshot=shots, nrec=24,
                      f_ref=25.0, v_pml=3300.0)
    q = oracle.make_problem(0, nz, nx, pml, 10.0, np.float32(1e-3), nt, shots, 24, 25.0,
                            v_pml=3300.0)
    t = [torch.tensor(x, device="cuda") for x in (v, w, src, rec, d_obs[:, None])]
    f64 = [x.astype(np.float64) for x in (v, w, d_obs)]
    # workspaces full of NaN: nothing may depend on what they held
    ws = [sweep.alloc_workspace(p, m) for m in range(3)]
    for x in ws:
        x.fill_(0xFF)
    d = sweep.sweep_forward(p, *t[:4], ws=ws[0]).cpu().numpy()[:, 0]
    assert rel(d, oracle.acoustic_forward(q, f64[0], f64[1], src, rec)) <= 1e-4
    g = sweep.sweep_adjoint(p, t[0], t[4], t[2], t[3], ws=ws[1]).cpu().numpy()
    assert rel(g, oracle.acoustic_adjoint(q, f64[0], f64[2], src, rec)) <= 1e-4
    g, j, il = sweep.sweep_gradient(p, *t, want_illum=True, ws=ws[2])
    ref, j_ref = oracle.acoustic_gradient(q, f64[0], f64[1], src, rec, f64[2])
    assert rel(g.cpu().numpy(), ref) <= 1e-3
    assert abs(j.item() - j_ref) <= 1e-4 * j_ref
    # the stencil + CPML kernels (deterministic mode) agree, illumination included
    p.flags |= sweep.F_DETERMINISTIC
    g2, _, il2 = sweep.sweep_gradient(p, *t, want_illum=True)
    assert rel(g.cpu(), g2.cpu()) <= 1e-4 and rel(il.cpu(), il2.cpu()) <= 1e-4
