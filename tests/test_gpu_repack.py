"""Ensembles that are rewritten into whole frame tiles before beamforming: every storage type,
frame counts around the edges of the tiles (8, 16 and 32 frames and their sums), 2D and 3D,
one and several transmits, against the FP64 oracle and the direct kernel."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2604_06257_gb300 as m
from metrics import nrmse_db

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def repack_small_grids():
    """These grids are too small for repacking to pay; test_gpu_repack_rule.py has the rule."""
    m.mach_debug_force_repack(True)
    yield
    m.mach_debug_force_repack(False)

CASES = [(F, dt) for F in (5, 8, 9, 16, 17, 25, 31, 32, 33, 40, 41, 49, 64, 65, 100)
         for dt in ("c64", "f16x2", "bf16x2", "c64split")
         if dt != "c64split" or (F % 4 == 0 and F not in (8, 16, 32, 64))]


def dense(F, dt, ndim=2, T=1):
    """Few samples and many voxels, so that repacking pays."""
    name = "doppler2d" if ndim == 2 else "volume3d"
    acq = synth.make_acquisition(name, "small")
    dims = (53, 1, 67) if ndim == 2 else (17, 13, 19)
    ang = np.zeros((T, 2))
    ang[:, 0] = np.linspace(-0.1, 0.1, T) if T > 1 else 0.0
    # a shallow grid under the middle of the array, so that 200 samples reach its floor
    mid = len(acq.elem_pos) // 2
    origin = (-dims[0] * 5e-5, 0.0 if ndim == 2 else -dims[1] * 5e-5, 1e-3)
    return acq.replace(grid_dims=dims, grid_origin=origin, grid_step=(1e-4, 0.0 if ndim == 2 else 1e-4, 1e-5),
                       elem_pos=acq.elem_pos[mid - 12:mid + 12], tx_angles=ang, n_samples=200, n_frames=F, iq_dtype=dt)


def stored(acq, seed):
    iq = synth.random_iq(acq.replace(iq_dtype="c64"), seed, device="cuda")
    x = synth.iqmod.to_c64split(iq) if acq.iq_dtype == "c64split" else synth.iqmod.to_storage(iq, acq.iq_dtype)
    ref = iq.cpu() if acq.iq_dtype in ("c64", "c64split") else synth.iqmod.from_storage(x.cpu())
    return x, ref


@pytest.mark.parametrize("F,dt", CASES)
def test_repacked_frames_match_oracle(F, dt):
    for ndim, T in ((2, 1), (2, 3), (3, 2)):
        acq = dense(F, dt, ndim, T)
        if acq.n_vox < 16 * acq.n_samples:
            pytest.fail("grid too small for the repacked route")
        x, ref = stored(acq, F + T)
        with m.Plan(**m.plan_kwargs(acq)) as p:
            assert "+x" in p.info()["variant"], p.info()
            pd, y = p.power_doppler(x, want_y=True)
            y_only = p.run(x)
            pd_only, _ = p.power_doppler(x)
            torch.cuda.synchronize()
            assert p.device_status() == m.MACH_OK
            # a captured run allocates nothing: it takes the direct kernel
            g = torch.cuda.CUDAGraph()
            yg = torch.zeros_like(y)
            with torch.cuda.graph(g):
                m.mach_das_run(p.handle, x, yg)
            g.replay()
            torch.cuda.synchronize()
        assert torch.equal(y, y_only) and torch.equal(pd, pd_only)
        idx = np.arange(0, acq.n_vox, 7)
        y_ref, pd_ref = oracle.das(acq, ref, idx)
        assert nrmse_db(y.cpu().numpy()[idx], y_ref) <= -100, (ndim, T)
        assert nrmse_db(pd.cpu().numpy()[idx].astype(np.float64), pd_ref) <= -100, (ndim, T)
        assert nrmse_db(yg.cpu().numpy(), y.cpu().numpy()) <= -110, (ndim, T)


def test_repacked_runs_share_a_plan_across_streams():
    """Concurrent calls on one plan take separate workspaces."""
    acq = dense(25, "f16x2", 2, 3)
    xs = [stored(acq, s)[0] for s in range(6)]
    with m.Plan(**m.plan_kwargs(acq)) as p:
        want = [p.run(x) for x in xs]
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in xs]
        got = [torch.zeros_like(w) for w in want]
        torch.cuda.synchronize()
        for _ in range(4):
            for s, x, y in zip(streams, xs, got):
                m.mach_das_run(p.handle, x, y, stream=s)
        torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dt", ["c64", "f16x2", "bf16x2"])
def test_batch_of_repacked_instances(dt):
    """A batch mixing every frame-tile shape (and channel lanes) in 2D and 3D; a captured run
    follows a later bind, also one that leaves out an instance's Power Doppler."""
    frames = [2, 5, 8, 13, 16, 20, 32, 33, 41, 49, 64, 25]
    acqs = [dense(F, dt, 2 + i % 2, 1 + i % 3) for i, F in enumerate(frames)]
    sets = [[stored(a, 100 * k + i)[0] for i, a in enumerate(acqs)] for k in range(2)]
    def out():
        return ([torch.zeros((a.n_vox, a.n_frames), dtype=torch.complex64, device="cuda") for a in acqs],
                [torch.zeros(a.n_vox, dtype=torch.float32, device="cuda") for a in acqs])
    with m.Batch([m.plan_kwargs(a) for a in acqs]) as b:
        y0, pd0 = out()
        b.bind(sets[0], y0, pd0)
        b.run()
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            b.run()
        y1, pd1 = out()
        b.bind(sets[1], y1, pd1[:-4] + [None] + pd1[-3:])
        g.replay()
        torch.cuda.synchronize()
    assert not pd1[-4].any()
    for xs, ys, pds in ((sets[0], y0, pd0), (sets[1], y1, pd1)):
        for i, (a, x, y, pd) in enumerate(zip(acqs, xs, ys, pds)):
            idx = np.arange(0, a.n_vox, 13)
            y_ref, pd_ref = oracle.das(a, synth.iqmod.from_storage(x.cpu()), idx)
            assert nrmse_db(y.cpu().numpy()[idx], y_ref) <= -100, i
            if pds is pd1 and i == len(acqs) - 4:
                continue
            assert nrmse_db(pd.cpu().numpy()[idx].astype(np.float64), pd_ref) <= -100, i


@pytest.mark.parametrize("F,direct", [(7, "frames_c64_scalar_ft32"), (25, "frames_c64_scalar_ft32"), (12, "frames_c64_ft16"),
                                      (70, "frames_c64_ft64")])
def test_nan_and_inf_samples_reach_only_kept_terms(F, direct):
    """The same frames of the same voxels are not finite as with the kernel that skips dropped
    terms."""
    acq = dense(F, "c64", 2, 2)
    x, _ = stored(acq, F)
    for k, bad in ((0, float("nan")), (11, float("inf")), (23, -float("inf"))):
        x[k % 2, k, 60 + k, (3 * k) % F] = bad
        x[1 - k % 2, k, 40, (5 * k) % F] = bad
    with m.Plan(**m.plan_kwargs(acq)) as p:
        assert "+x" in p.info()["variant"]
        y = p.run(x)
    m.mach_debug_force_variant(direct)
    try:
        with m.Plan(**m.plan_kwargs(acq)) as p:
            ref = p.run(x)
    finally:
        m.mach_debug_force_variant(None)
    torch.cuda.synchronize()
    ok = torch.isfinite(torch.view_as_real(ref)).all(-1)
    assert bool(ok.any()) and not bool(ok.all())
    assert torch.equal(torch.isfinite(torch.view_as_real(y)).all(-1), ok)


def batch_and_plans(acqs, xs):
    """(batch frames, single plans' frames, those with the kernels that read the ensembles directly);
    checks that the batch has other items than its lane mappings would."""
    ys = [torch.zeros((a.n_vox, a.n_frames), dtype=torch.complex64, device="cuda") for a in acqs]
    with m.Batch([m.plan_kwargs(a) for a in acqs]) as b:
        b.bind(xs, ys, None)
        b.run()
        torch.cuda.synchronize()
        info = b.info()
    with m.Batch([m.plan_kwargs(a) for a in acqs], shapes=[(s[0], s[1], None) for s in info["shapes"]]) as b:
        assert b.info()["items"] != info["items"]
    plans, direct = [], []
    for a, x in zip(acqs, xs):
        with m.Plan(**m.plan_kwargs(a)) as p:
            name = p.info()["variant"]
            plans.append(p.run(x))
        m.mach_debug_force_variant(name.split("+")[0])
        try:
            with m.Plan(**m.plan_kwargs(a)) as p:
                direct.append(p.run(x))
        finally:
            m.mach_debug_force_variant(None)
        assert ("+x" in name) == (a.n_frames > 4)
    torch.cuda.synchronize()
    return ys, plans, direct


def test_batch_instances_are_repacked():
    """Bit for bit the frames of a repacking plan, which differ from those of the direct kernels where
    several transmits are summed in another order; the 73 instances with a 32-frame tile
    exceed one launch's entries."""
    frames = [25, 32, 27, 31] * 18 + [41, 5, 16, 2, 13]
    acqs = [dense(F, "c64", 2 + (i // 4) % 2, 1 + i % 2) for i, F in enumerate(frames)]
    xs = [stored(a, i)[0] for i, a in enumerate(acqs)]
    ys, plans, direct = batch_and_plans(acqs, xs)
    for a, y, p, d in zip(acqs, ys, plans, direct):
        assert torch.equal(y, p)
        assert nrmse_db(y.cpu().numpy(), d.cpu().numpy()) <= -110
    assert sum(not torch.equal(y, d) for y, d in zip(ys, direct)) >= 10


def test_batch_repacks_up_to_its_budget():
    """Two instances (of the same IQ) whose workspaces together exceed a sixteenth of the device's
    memory: the first is repacked, the second beamformed by a lane mapping."""
    total = torch.cuda.mem_get_info()[1]
    acq = dense(64, "c64", 3, 2)
    C = int(0.6 * total / 16 / (2 * acq.n_samples * 64 * 8))      # elements that fill 0.6 of it
    e = np.zeros((C, 3), np.float32)
    e[:, 0], e[:, 1] = np.linspace(-4e-3, 4e-3, C), np.linspace(-1e-3, 1e-3, C)
    acq = acq.replace(elem_pos=e)
    x = torch.view_as_complex(torch.randn((2, C, acq.n_samples, 64, 2), device="cuda"))
    ys = [torch.zeros((acq.n_vox, 64), dtype=torch.complex64, device="cuda") for _ in range(2)]
    with m.Batch([m.plan_kwargs(acq)] * 2) as b:
        b.bind([x, x], ys, None)
        b.run()
        torch.cuda.synchronize()
    with m.Plan(**m.plan_kwargs(acq)) as p:
        assert "+x32" in p.info()["variant"]
        y = p.run(x)
        torch.cuda.synchronize()
    assert torch.equal(ys[0], y) and not torch.equal(ys[1], y)
    assert nrmse_db(ys[1].cpu().numpy(), y.cpu().numpy()) <= -100
