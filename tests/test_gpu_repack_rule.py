"""When an ensemble is repacked: only where that was measured faster than the kernel that reads
it directly.  Grids on both sides of every line of the rule; the direct side slowed down to half
its speed when it was repacked."""
import numpy as np
import pytest
import torch

import synth
import paper_2604_06257_gb300 as m
from metrics import nrmse_db

pytestmark = pytest.mark.gpu


def grid(side, F, dt, f_number, T, S, ndim=2, elems=128):
    """side^ndim points 0.1 mm apart, 5 mm below a 0.3 mm pitch array."""
    acq = synth.make_acquisition("doppler2d" if ndim == 2 else "volume3d", "small")
    n = elems if ndim == 2 else int(np.sqrt(elems))
    at = (np.arange(n) - (n - 1) / 2) * 0.3e-3
    x, y = (at, np.zeros(n)) if ndim == 2 else (a.ravel() for a in np.meshgrid(at, at))
    ang = np.zeros((T, 2))
    ang[:, 0] = np.linspace(-0.17, 0.17, T) if T > 1 else 0.0
    half = -(side - 1) * 0.5e-4
    return acq.replace(elem_pos=np.stack([x, y, 0 * x], 1).astype(np.float32), tx_angles=ang, f_number=f_number,
                       apod="boxcar", n_samples=S, n_frames=F, iq_dtype=dt, t0=0.0,
                       grid_dims=(side, side if ndim == 3 else 1, side),
                       grid_origin=(half, half if ndim == 3 else 0.0, 5e-3), grid_step=(1e-4, 1e-4 if ndim == 3 else 0.0, 1e-4))


DIRECT = [  # repacked, these took 1.1 to 2 times as long
    (128, 40, "c64split", 1.0, 1, 585), (128, 40, "c64", 1.0, 1, 585), (96, 48, "f16x2", 1.0, 3, 486), (128, 64, "f16x2", 3.0, 1, 585),
    (40, 64, "c64", 3.0, 1, 452, 3, 576), (256, 64, "bf16x2", 3.0, 9, 983), (48, 20, "c64", 3.0, 3, 135), (48, 32, "bf16x2", 3.0, 3, 135),
    (128, 20, "f16x2", 3.0, 1, 585)]
REPACKED = [
    (48, 5, "c64", 3.0, 1, 135), (48, 33, "c64", 1.0, 1, 135), (64, 12, "c64split", 3.0, 1, 240), (128, 20, "c64", 1.0, 1, 585),
    (128, 28, "c64split", 1.0, 3, 585), (192, 20, "f16x2", 1.0, 3, 784), (256, 40, "c64", 1.0, 3, 983), (256, 64, "f16x2", 1.0, 3, 983),
    (64, 72, "c64", 1.0, 1, 240), (144, 20, "f16x2", 1.0, 1, 518, 2, 240), (144, 24, "bf16x2", 1.0, 1, 518, 2, 240),
    (256, 28, "c64split", 3.0, 3, 983)]


@pytest.mark.parametrize("case", DIRECT)
def test_small_or_narrow_grids_stay_on_their_kernel(case):
    with m.Plan(**m.plan_kwargs(grid(*case))) as p:
        info = p.info()
    assert "+x" not in info["variant"], info


@pytest.mark.parametrize("case", REPACKED)
def test_dense_grids_are_repacked(case):
    with m.Plan(**m.plan_kwargs(grid(*case))) as p:
        info = p.info()
    assert "+x" in info["variant"], info


def test_either_route_gives_the_same_frames():
    acq = grid(128, 40, "c64split", 1.0, 1, 585)
    x = synth.iqmod.to_c64split(synth.random_iq(acq.replace(iq_dtype="c64"), 3, device="cuda"))
    with m.Plan(**m.plan_kwargs(acq)) as p:
        pd, y = p.power_doppler(x, want_y=True)
    m.mach_debug_force_repack(True)
    try:
        with m.Plan(**m.plan_kwargs(acq)) as p:
            assert "+x" in p.info()["variant"]
            pd_r, y_r = p.power_doppler(x, want_y=True)
    finally:
        m.mach_debug_force_repack(False)
    torch.cuda.synchronize()
    assert nrmse_db(y_r.cpu().numpy(), y.cpu().numpy()) <= -110
    assert nrmse_db(pd_r.cpu().numpy().astype(np.float64), pd.cpu().numpy().astype(np.float64)) <= -110


def batch_items(acqs):
    """Items of the default batch, of its lane mappings, and with everything repacked."""
    kws = [m.plan_kwargs(a) for a in acqs]
    with m.Batch(kws) as b:
        info = b.info()
    with m.Batch(kws, shapes=[(s[0], s[1], None) for s in info["shapes"]]) as b:
        lanes = b.info()["items"]
    m.mach_debug_force_repack(True)
    try:
        with m.Batch(kws) as b:
            repacked = b.info()["items"]
    finally:
        m.mach_debug_force_repack(False)
    assert lanes != repacked
    return info["items"], lanes, repacked


def test_batches_of_small_instances_stay_in_one_launch():
    """Many small instances run in the persistent launch: repacked one after another they took two to eight
    times as long.  A few, larger ones, and small ones that are dear on lanes are repacked."""
    small = grid(64, 25, "f16x2", 1.5, 1, 248)
    large = grid(40, 28, "f16x2", 1.0, 3, 452, 3, 576)
    for acqs, repacked in (([small], True), ([small] * 12, False), ([small] * 30, False), ([large] * 2, True),
                           ([grid(128, 25, "f16x2", 1.0, 3, 585)] * 6, True), ([grid(28, 16, "c64", 3.0, 1, 423, 3, 256)] * 12, True)):
        items, lanes, all_repacked = batch_items(acqs)
        assert items == (all_repacked if repacked else lanes), len(acqs)
    items, lanes, all_repacked = batch_items([small] * 12 + [large])
    assert items not in (lanes, all_repacked)         # the large one alone
