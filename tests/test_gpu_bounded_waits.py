"""Waits that run out while copies are in flight (a limit of one poll, nothing stalled): the kernels
report a timeout or finish, their blocks leave after their own copies have landed, and
the next call is right."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2604_06257_gb300 as m
from metrics import nrmse_db
from paper_2604_06257_gb300 import nn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,dt,repack", [(32, "c64split", False), (64, "c64split", False), (30, "c64", False), (25, "c64", True)])
def test_beamforming(F, dt, repack):
    acq = synth.make_acquisition("doppler2d", "small").replace(
        grid_dims=(96, 1, 96), grid_origin=(-4.8e-3, 0.0, 5e-3), grid_step=(1e-4, 0.0, 1e-4), n_samples=460, n_frames=F, iq_dtype=dt)
    iq = synth.random_iq(acq.replace(iq_dtype="c64"), F, device="cuda")
    x = synth.iqmod.to_c64split(iq) if dt == "c64split" else iq
    kw = m.plan_kwargs(acq)
    m.mach_debug_force_repack(repack)
    if dt == "c64" and not repack:
        m.mach_debug_force_variant("staged_c64_ft32_v4w7")
    m.mach_debug_set_wait_limit(1)
    try:
        with m.Plan(**kw) as p:
            assert ("+x" in p.info()["variant"]) == repack
            for _ in range(4):
                p.power_doppler(x, want_y=True)
            assert p.device_status() in (m.MACH_OK, m.MACH_ERR_TIMEOUT)
        m.mach_debug_force_variant(None)
        if not repack and dt == "c64":
            with m.Batch([kw] * 6, shapes=[(2, 8, None)] * 6) as b:
                ys = [torch.zeros((acq.n_vox, F), dtype=torch.complex64, device="cuda") for _ in range(6)]
                b.bind([x] * 6, ys, None)
                for _ in range(4):
                    b.run()
                torch.cuda.synchronize()
    finally:
        m.mach_debug_set_wait_limit(0)
        m.mach_debug_force_repack(False)
        m.mach_debug_force_variant(None)
    with m.Plan(**kw) as p:
        pd, y = p.power_doppler(x, want_y=True)
        assert p.device_status() == m.MACH_OK
    idx = np.arange(0, acq.n_vox, 13)
    assert nrmse_db(y.cpu().numpy()[idx], oracle.das(acq, iq.cpu(), idx)[0]) <= -100


@pytest.mark.parametrize("ci,co", [(16, 16), (32, 32), (64, 128), (128, 256)])
def test_convolutions(ci, co):
    gen = torch.Generator(device="cuda").manual_seed(ci + co)
    shape = (2, 9, 33, 40)
    x = torch.randn(shape + (ci,), device="cuda", generator=gen).to(torch.bfloat16)
    g = torch.randn(shape + (co,), device="cuda", generator=gen).to(torch.bfloat16)
    w = torch.randn((27, ci, co), device="cuda", generator=gen) * 0.05
    pk, pkt = nn.mach_nn_pack_weights(w, ci, co)

    def both():
        y = torch.zeros(shape + (co,), device="cuda", dtype=torch.bfloat16)
        dx = torch.zeros(shape + (ci,), device="cuda", dtype=torch.bfloat16)
        dw = torch.zeros((27, ci, co), device="cuda")
        nn.mach_nn_conv3d_tc(x, pk, co, None, y, None)
        nn.mach_nn_conv3d_tc(g, pkt, ci, None, dx, None, flip=True)
        nn.mach_nn_conv3d_wgrad(x, g, dw)
        return y, dx, dw

    want = both()
    assert nn.mach_nn_device_status() == m.MACH_OK
    nn.mach_nn_debug_conv(False, 1)
    try:
        for _ in range(4):
            both()
        assert nn.mach_nn_device_status() in (m.MACH_OK, m.MACH_ERR_TIMEOUT)
    finally:
        nn.mach_nn_debug_conv(False, 0)
    got = both()
    assert nn.mach_nn_device_status() == m.MACH_OK
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    # the blocks' float32 atomics come in any order
    assert float((got[2] - want[2]).norm() / want[2].norm()) < 1e-5
