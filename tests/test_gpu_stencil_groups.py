"""The forward stencil kernel with two groups of warps per CTA (more than about
two units a CTA) against the same kernel with one.

Three problems of 180, 144 and 132 units (at 132 to 152 SMs one each, so one group
alone) share the launches of a batch (three units a CTA: two groups, an odd count).
In the deterministic mode every cell is written once per step, so the traces are the
same to the last bit, with 32-row and with 16-row tiles.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows16", [False, True])
def test_batch_equals_single_runs(rows16):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14189_gb300 import inputs, sweep
    flags = sweep.F_DETERMINISTIC | (sweep.F_ROWS16 if rows16 else 0)
    nt, rng, args = 25, np.random.default_rng(3), []
    for nz, nx, pml, shots in [(70, 300, 10, 20), (60, 200, 12, 24), (40, 120, 5, 33)]:
        v = (2000 + 500 * rng.random((nz, nx))).astype(np.float32)
        src = np.stack([rng.integers(0, nz, shots), rng.integers(0, nx, shots)], -1)
        rec = np.stack([rng.integers(0, nz, (shots, 31)), rng.integers(0, nx, (shots, 31))], -1)
        p = sweep.problem(nz=nz, nx=nx, pml=pml, dx=10.0, dt=1e-3, nt=nt, nshot=shots, nrec=31,
                          f_ref=25.0, flags=flags)
        w = np.stack([inputs.ricker(40.0, 1e-3, nt)] * shots).astype(np.float32)
        args.append((p, torch.tensor(v).cuda(), torch.tensor(w).cuda(),
                     torch.tensor(src.astype(np.int32)).cuda(),
                     torch.tensor(rec.astype(np.int32)).cuda()))
    batch = sweep.sweep_forward_batch(*[list(x) for x in zip(*args)])
    for a, d in zip(args, batch):
        one = sweep.sweep_forward(*a)
        assert one.abs().max() > 0
        assert torch.equal(one, d)
