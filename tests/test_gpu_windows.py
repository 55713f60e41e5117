"""Delays far larger than the record (a distant grid whose recording starts late: receive and
transmit delay nearly cancel): a staged window's float32 bounds may then miss a kept term, so
plans keep the kernels that look for its taps in global memory, and repack nothing."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2604_06257_gb300 as m
from metrics import nrmse_db

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def repack_wherever_the_kernels_can():
    m.mach_debug_force_repack(True)
    yield
    m.mach_debug_force_repack(False)

S, REACH = 200, 2.0 ** 26            # samples a record, samples of receive delay
EDGE = 24                            # more rows than 4.5 units of 2^-24 of REACH


def distant(F, dt):
    """53 x 67 px at 45 degrees and REACH samples from 24 elements."""
    acq = synth.make_acquisition("doppler2d", "small")
    k = acq.fs / acq.c
    mid = len(acq.elem_pos) // 2
    x0, z0 = 0.6 * REACH / k, 0.8 * REACH / k
    t0 = (z0 + float(np.hypot(x0, z0))) / acq.c - 0.5 * S / acq.fs     # mid-record at the corner
    return acq.replace(grid_dims=(53, 1, 67), grid_origin=(x0, 0.0, z0), grid_step=(1e-4, 0.0, 1e-4), t0=t0,
                       elem_pos=acq.elem_pos[mid - 12:mid + 12], tx_angles=np.zeros((1, 2)), n_samples=S,
                       n_frames=F, iq_dtype=dt, apod="none")


def stored(acq, seed):
    """Random IQ, nothing at the record's ends: a window wholly beyond them is not staged."""
    iq = synth.random_iq(acq.replace(iq_dtype="c64"), seed, device="cuda")
    iq[:, :, :EDGE] = 0
    iq[:, :, S - EDGE:] = 0
    x = synth.iqmod.to_c64split(iq) if acq.iq_dtype == "c64split" else synth.iqmod.to_storage(iq, acq.iq_dtype)
    return x, iq.cpu() if acq.iq_dtype in ("c64", "c64split") else synth.iqmod.from_storage(x.cpu())


def check(acq, ref, y, pd):
    y_ref, pd_ref = oracle.das(acq, ref)
    assert np.abs(y_ref).max() > 0
    assert nrmse_db(y.cpu().numpy(), y_ref) <= -100
    assert nrmse_db(pd.cpu().numpy().astype(np.float64), pd_ref) <= -100


def test_terms_outside_their_windows():
    repackable = [distant(F, dt) for F, dt in ((25, "c64"), (16, "c64"), (20, "f16x2"), (9, "bf16x2"), (40, "c64split"))]
    for acq in repackable:           # before anything runs: no plan may trust its windows here
        with m.Plan(**m.plan_kwargs(acq)) as p:
            assert "+x" not in p.info()["variant"], p.info()
    for acq in repackable + [distant(F, "c64split") for F in (8, 16, 32, 64)]:
        x, ref = stored(acq, acq.n_frames)
        with m.Plan(**m.plan_kwargs(acq)) as p:
            pd, y = p.power_doppler(x, want_y=True)
            torch.cuda.synchronize()
            assert p.device_status() == m.MACH_OK
        check(acq, ref, y, pd)


def test_batch_terms_outside_their_windows():
    acqs = [distant(F, "c64") for F in (2, 16, 25, 32)]
    with m.Plan(**m.plan_kwargs(acqs[2])) as p:
        assert "+x" not in p.info()["variant"], p.info()
    sets = [stored(a, i) for i, a in enumerate(acqs)]
    ys = [torch.zeros((a.n_vox, a.n_frames), dtype=torch.complex64, device="cuda") for a in acqs]
    pds = [torch.zeros(a.n_vox, dtype=torch.float32, device="cuda") for a in acqs]
    with m.Batch([m.plan_kwargs(a) for a in acqs]) as b:
        b.bind([x for x, _ in sets], ys, pds)
        b.run()
        torch.cuda.synchronize()
    for a, (_, ref), y, pd in zip(acqs, sets, ys, pds):
        check(a, ref, y, pd)
