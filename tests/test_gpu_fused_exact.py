"""Fused acoustic kernels against the stencil and CPML kernels, to the last bit.

Both round every product and sum alike, so they may differ only where the per-step
kernels leave the order of two additions open: in a corner of the border (the two
axes' CPML terms) and at a receiver within 4 cells of the border (the residual).
Here no wave meets either: without a border; or with sources and receivers around
the middle of each side of a square, receivers 6 cells inside it, and fewer steps
than a wave (4 cells a step, from a source forward and from a receiver backward)
takes to a corner or the 4 cells around it.  A batch of one problem runs the per-step kernels; the
illumination, which a batch does not give, is the deterministic mode's.

1, 2 and 3 shots on a padded 280 x 280 grid and 1 on 310 x 310 are 144, 288, 432
and 169 tiles of 24 x 24: at 152 SMs each of the four launch variants, forward and
backward.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# (cells a side, border, steps, shots)
CASES = [(240, 20, 27, 1), (240, 20, 27, 2), (240, 20, 27, 3), (270, 20, 30, 1), (250, 3, 28, 1),
         (200, 0, 61, 1), (150, 0, 50, 3)]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_fused_equals_per_step(case):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14189_gb300 import inputs, sweep
    n, pml, nt, shots = case
    rng = np.random.default_rng(sum(case))
    # along the middle of each side: first coordinate across it, second along it
    near = n // 2 + (np.arange(-7, 8) if pml else rng.permutation(n)[:15] - n // 2)
    if pml:
        assert min(near.min(), n - 1 - near.max()) - 3 > 4 * nt
    sides = [np.stack(s, -1) for s in ((0 * near + 6, near), (near, 0 * near + n - 7),
                                      (0 * near + n - 7, near), (near, 0 * near + 6))]
    rec = np.stack([np.concatenate(sides)] * shots).astype(np.int32)
    src = np.stack([sides[(i + pml) % 4][7] for i in range(shots)]).astype(np.int32)
    src = np.where(src == 6, 1, np.where(src == n - 7, n - 2, src)).astype(np.int32)
    v = np.clip(2400 + 300 * rng.standard_normal((n, n)), 1500, 3300).astype(np.float32)
    w = np.stack([inputs.ricker(40.0, 1e-3, nt)] * shots).astype(np.float32)
    d_obs = (0.01 * rng.standard_normal((shots, 1, rec.shape[1], nt))).astype(np.float32)
    t = [torch.tensor(x, device="cuda") for x in (v, w, src, rec, d_obs)]
    p = sweep.problem(nz=n, nx=n, pml=pml, dx=10.0, dt=1e-3, nt=nt, nshot=shots,
                      nrec=rec.shape[1], f_ref=25.0, v_pml=3300.0)
    before = sweep.kernel_launches()
    d = sweep.sweep_forward(p, *t[:4])
    assert sweep.kernel_launches() - before < nt  # (two a step without the fused kernels)
    d1 = sweep.sweep_forward_batch([p], *[[x] for x in t[:4]])[0]
    assert d.abs().max() > 0 and torch.equal(d, d1)
    g, j, il = sweep.sweep_gradient(p, *t, want_illum=True)
    (g1,), (j1,) = sweep.sweep_gradient_batch([p], *[[x] for x in t])
    assert g.abs().max() > 0 and torch.equal(g, g1)
    assert j.item() == j1.item()
    p.flags |= sweep.F_DETERMINISTIC
    _, j2, il2 = sweep.sweep_gradient(p, *t, want_illum=True)
    assert torch.equal(il, il2) and j.item() == j2.item()
