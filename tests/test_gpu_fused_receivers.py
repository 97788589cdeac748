"""Fused acoustic kernels with so many receivers a shot that shared memory decides
which variant can run: a CTA lists them all (8 bytes each, backward 4 more a step).

The two-step 32 x 32 backward variant has room for 1631 (it serves one shot on a
padded 336 x 336 or 64 x 2020 grid at 152 SMs), three CTAs of the 16 x 32 one for
1748 each and two of the one-step 32 x 32 one for 1833; 2048 is the most of any.
At each limit and past it, against the FP64 oracle, with the suite's tolerances
for adjoint sources and seismograms (1e-4 relative L2) and gradients (1e-3).
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

# (nz, nx, pml, steps, shots or shots per SM, receivers)
CASES = [(256, 256, 40, 15, 1, n) for n in (1631, 1632, 2048, 2049)] + [
    (44, 2000, 10, 12, 1, 2000), (12, 12, 6, 9, 1.5, 1748), (12, 12, 6, 9, 1.5, 1749),
    (12, 12, 6, 9, 2.0, 1833), (12, 12, 6, 9, 2.0, 1834)]


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("case", CASES, ids=str)
def test_many_receivers(case):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14189_gb300 import inputs, sweep
    nz, nx, pml, nt, shots, nrec = case
    if shots != 1:
        shots = int(shots * torch.cuda.get_device_properties(0).multi_processor_count)
    rng = np.random.default_rng(nrec + nz)
    v = np.clip(2200 + 300 * rng.standard_normal((nz, nx)), 1500, 3300).astype(np.float32)
    src = np.stack([rng.integers(0, nz, shots), rng.integers(0, nx, shots)], -1).astype(np.int32)
    rec = np.stack([rng.integers(0, nz, (shots, nrec)), rng.integers(0, nx, (shots, nrec))],
                   -1).astype(np.int32)
    rec[:, :64] = src[:, None] + np.clip(rng.integers(-4, 5, (shots, 64, 2)), -src[:, None],
                                         np.array([nz - 1, nx - 1]) - src[:, None])
    w = np.stack([inputs.ricker(60.0, 1e-3, nt)] * shots).astype(np.float32)
    d_obs = rng.standard_normal((shots, nrec, nt)).astype(np.float32)
    t = [torch.tensor(x, device="cuda") for x in (v, w, src, rec, d_obs[:, None])]
    f64 = [x.astype(np.float64) for x in (v, w, d_obs)]
    p = sweep.problem(nz=nz, nx=nx, pml=pml, dx=10.0, dt=1e-3, nt=nt, nshot=shots, nrec=nrec,
                      f_ref=25.0, v_pml=3300.0)
    q = oracle.make_problem(0, nz, nx, pml, 10.0, np.float32(1e-3), nt, shots, nrec, 25.0,
                            v_pml=3300.0)
    d = sweep.sweep_forward(p, *t[:4]).cpu().numpy()[:, 0]
    assert rel(d, oracle.acoustic_forward(q, f64[0], f64[1], src, rec)) <= 1e-4
    a = sweep.sweep_adjoint(p, t[0], t[4], t[2], t[3]).cpu().numpy()
    assert rel(a, oracle.acoustic_adjoint(q, f64[0], f64[2], src, rec)) <= 1e-4
    g, j, _ = sweep.sweep_gradient(p, *t)
    ref, j_ref = oracle.acoustic_gradient(q, f64[0], f64[1], src, rec, f64[2])
    assert rel(g.cpu().numpy(), ref) <= 1e-3
    assert abs(j.item() - j_ref) <= 1e-4 * j_ref
