"""Every launch variant of the fused acoustic kernels, and the per-step kernels
beyond them, against the FP64 oracle: forward, adjoint and gradient.

The rule that picks a variant counts tiles against the GPU's SMs, so the shot
counts come from them.  It is written down here once more; the number of kernels
that a call launches says which of them ran (3, 2 or 1 steps a launch, two
launches a step otherwise).  Tolerances are the suite's: 1e-4 relative L2 for
seismograms, adjoint sources and the misfit, 1e-3 for gradients.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

# (steps a launch, tile rows, tile columns, CTAs per SM, waves in a gradient,
# most tiles of a shot outside of a gradient)
ANY = 1 << 40
FORWARD = [(3, 24, 24, 1, 1, ANY), (2, 32, 32, 1, 1, ANY), (2, 24, 24, 2, 1, ANY),
           (2, 24, 24, 3, 2, ANY)]
BACKWARD = [(2, 24, 24, 1, 1, ANY), (2, 32, 32, 1, 1, ANY), (1, 16, 32, 3, 1, ANY),
            (1, 32, 32, 2, 1, 16)]

# (nz, nx, pml), shots a SM (rounded up), and shots more
CASES = [((12, 12, 6), 0.0, 3), ((17, 17, 6), 0.5, 1), ((12, 12, 6), 1.0, 1),
         ((12, 12, 6), 2.0, 0), ((12, 12, 6), 2.0, 1), ((12, 12, 6), 6.0, 0),
         ((12, 12, 6), 6.0, 1), ((130, 100, 10), 0.0, 12), ((110, 90, 5), 0.0, 16)]
CASE_IDS = [f"{c[0]}-{c[1]}x-{c[2]}" for c in CASES]


def variant(table, grid, shots, sms, gradient):
    """Index in the table, or None: the per-step kernels."""
    nz, nx, pml = grid
    for i, (_, bz, bx, res, waves, alone) in enumerate(table):
        tiles = -(-(nz + 2 * pml) // bz) * -(-(nx + 2 * pml) // bx)
        if not gradient and tiles > alone:
            continue
        if tiles * shots <= sms * res * (waves if gradient else 1):
            return i
    return None


def launches(table, v, steps):
    return 2 * steps if v is None else -(-steps // table[v][0])


def choices(case, sms):
    grid, per_sm, more = case
    shots = int(np.ceil(per_sm * sms)) + more
    return shots, [variant(t, grid, shots, sms, g) for t, g in
                   ((FORWARD, False), (BACKWARD, False), (FORWARD, True), (BACKWARD, True))]


def test_the_cases_cover_the_variants():
    """On GPUs of 132 to 152 SMs every entry of both tables and the per-step
    kernels are reached, alone and in a gradient."""
    for sms in (132, 148, 152):
        got = [set() for _ in range(4)]
        for c in CASES:
            for s, v in zip(got, choices(c, sms)[1]):
                s.add(v)
        assert all(s == {None, 0, 1, 2, 3} for s in got), (sms, got)


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("case", CASES, ids=CASE_IDS)
def test_variant_matches_oracle(case):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14189_gb300 import inputs, sweep
    (nz, nx, pml), nt, nrec = case[0], 37, 9
    shots, (f, b, fg, bg) = choices(
        case, torch.cuda.get_device_properties(0).multi_processor_count)
    rng = np.random.default_rng(shots + nz)
    v = np.clip(2200 + 300 * rng.standard_normal((nz, nx)), 1500, 3300).astype(np.float32)
    src = np.stack([rng.integers(0, nz, shots), rng.integers(0, nx, shots)], -1).astype(np.int32)
    rec = np.stack([rng.integers(0, nz, (shots, nrec)), rng.integers(0, nx, (shots, nrec))],
                   -1).astype(np.int32)
    rec[:, 0], rec[:, 1] = (0, nx - 1), src  # a corner, and where the wave is
    w = np.stack([inputs.ricker(30.0, 1e-3, nt)] * shots).astype(np.float32)
    d_obs = (0.01 * rng.standard_normal((shots, nrec, nt))).astype(np.float32)
    t = [torch.tensor(x, device="cuda") for x in (v, w, src, rec, d_obs[:, None])]
    f64 = [x.astype(np.float64) for x in (v, w, d_obs)]
    p = sweep.problem(nz=nz, nx=nx, pml=pml, dx=10.0, dt=1e-3, nt=nt, nshot=shots, nrec=nrec,
                      f_ref=25.0, v_pml=3300.0)
    q = oracle.make_problem(0, nz, nx, pml, 10.0, np.float32(1e-3), nt, shots, nrec, 25.0,
                            v_pml=3300.0)
    n = [sweep.kernel_launches()]
    d = sweep.sweep_forward(p, *t[:4])
    n.append(sweep.kernel_launches())
    a = sweep.sweep_adjoint(p, t[0], t[4], t[2], t[3])
    n.append(sweep.kernel_launches())
    g, j, _ = sweep.sweep_gradient(p, *t)
    n.append(sweep.kernel_launches())
    # two set-up kernels a call; a gradient's residual, misfit and shot sum
    back = 2 * nt + 1  # per step: the last step has no CPML kernel
    assert n[1] - n[0] == 2 + launches(FORWARD, f, nt)
    if b is not None:  # (the per-step adjoint may launch a receiver listing too)
        assert n[2] - n[1] == 2 + launches(BACKWARD, b, nt + 1)
    else:
        assert n[2] - n[1] >= 2 + back
    if bg is not None:
        assert n[3] - n[2] == 5 + launches(FORWARD, fg, nt) + launches(BACKWARD, bg, nt + 1)
    else:
        assert n[3] - n[2] >= 5 + launches(FORWARD, fg, nt) + back
    assert rel(d.cpu().numpy()[:, 0], oracle.acoustic_forward(q, *f64[:2], src, rec)) <= 1e-4
    assert rel(a.cpu().numpy(), oracle.acoustic_adjoint(q, f64[0], f64[2], src, rec)) <= 1e-4
    ref, j_ref = oracle.acoustic_gradient(q, f64[0], f64[1], src, rec, f64[2])
    assert rel(g.cpu().numpy(), ref) <= 1e-3
    assert abs(j.item() - j_ref) <= 1e-4 * j_ref
