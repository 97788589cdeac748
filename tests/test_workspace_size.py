"""The size of a workspace: the same whatever the flags, and never smaller for a
larger problem, although the fused kernels, which only small problems without the
deterministic and one-launch flags run, need a second copy of the state."""
import numpy as np
import pytest
import torch

MODES = (0, 1, 2)


def problem(flags=0, **kw):
    from paper_2604_14189_gb300 import sweep
    a = dict(nz=8, nx=9, pml=4, dx=10.0, dt=1e-3, nt=7, nshot=2, nrec=3, f_ref=10.0,
             v_pml=3000.0)
    a.update(kw)
    return sweep.problem(flags=flags, **a)


@pytest.mark.parametrize("nshot", [1, 3, 4, 1000])
@pytest.mark.parametrize("n", [8, 16, 24, 200])
def test_size_ignores_the_flags(n, nshot):
    from paper_2604_14189_gb300 import sweep
    for mode in MODES:
        for flags in (sweep.F_DETERMINISTIC, sweep.F_ONE_LAUNCH, sweep.F_ROWS16,
                      sweep.F_RESIDUAL_IN):
            assert (sweep.workspace_bytes(problem(flags, nz=n, nx=n, nshot=nshot), mode)
                    == sweep.workspace_bytes(problem(nz=n, nx=n, nshot=nshot), mode))


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("field", ["nz", "nx", "pml", "nshot", "nrec", "nt"])
def test_size_grows_with_the_problem(field, mode):
    from paper_2604_14189_gb300 import sweep
    values = list(range(1, 70)) + [100, 150, 250, 400, 456, 457, 600, 912, 913, 2048, 2049]
    for nshot in (1, 60):
        size = [sweep.workspace_bytes(problem(**{"nshot": nshot, field: k}), mode)
                for k in values]
        assert all(b >= a > 0 for a, b in zip(size, size[1:]))


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.gpu
@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("tiles", [0.5, 3.0, 6.0])
def test_one_for_more_shots_is_enough(mode, tiles):
    """From `tiles` times the SMs on, in shots of one 24 x 24 tile, a problem takes
    the workspace of one with a shot more; so at 3 and 6 the larger problem
    runs the per-step kernels, alone and in a gradient.  The same kernels run in
    either workspace: FP32 rounding (a receiver's additions), 1e-5."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14189_gb300 import inputs, sweep
    n, nt, nrec = 12, 30, 5
    shots = int(tiles * torch.cuda.get_device_properties(0).multi_processor_count)
    kw = dict(nz=n, nx=n, pml=6, nt=nt, nrec=nrec)
    p, larger = problem(nshot=shots, **kw), problem(nshot=shots + 1, **kw)
    rng = np.random.default_rng(mode)
    t = [torch.tensor(x, device="cuda") for x in (
        (2200 + 300 * rng.random((n, n))).astype(np.float32),
        np.stack([inputs.ricker(30.0, 1e-3, nt)] * shots).astype(np.float32),
        rng.integers(0, n, (shots, 2)).astype(np.int32),
        rng.integers(0, n, (shots, nrec, 2)).astype(np.int32),
        rng.standard_normal((shots, 1, nrec, nt)).astype(np.float32))]

    def call(ws):
        if mode == 0:
            return sweep.sweep_forward(p, *t[:4], ws=ws)
        if mode == 1:
            return sweep.sweep_adjoint(p, t[0], t[4], t[2], t[3], ws=ws)
        return sweep.sweep_gradient(p, *t, ws=ws)[0]
    own = sweep.alloc_workspace(p, mode)
    assert rel(call(sweep.alloc_workspace(larger, mode)), call(own)) <= 1e-5
    with pytest.raises(sweep.SweepError) as e:
        call(own[:-256])
    assert e.value.code == sweep.EWORKSPACE
