"""Ensembles of one to four frames (element slices over the warps of a block): frame counts and
storage types, fewer elements than slices, ragged grids, y without Power Doppler and the
reverse, against the oracle and the 16-lane kernel."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2604_06257_gb300 as m
from metrics import nrmse_db

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [1, 2, 3, 4])
@pytest.mark.parametrize("dt", ["c64", "f16x2", "bf16x2"])
@pytest.mark.parametrize("name,elems", [("doppler2d", 5), ("doppler2d", 61), ("volume3d", 9)])
def test_short_ensembles(F, dt, name, elems):
    acq = synth.make_acquisition(name, "small")
    mid = len(acq.elem_pos) // 2
    acq = acq.replace(elem_pos=acq.elem_pos[mid - elems // 2:mid - elems // 2 + elems], n_frames=F, iq_dtype=dt)
    iq = synth.random_iq(acq.replace(iq_dtype="c64"), 10 * F + elems, device="cuda")
    x = synth.iqmod.to_storage(iq, dt)
    with m.Plan(**m.plan_kwargs(acq)) as p:
        assert "channels" in p.info()["variant"]
        pd, y = p.power_doppler(x, want_y=True)
        pd_only, _ = p.power_doppler(x)
        y_only = p.run(x)
        torch.cuda.synchronize()
    assert torch.equal(y, y_only) and torch.equal(pd, pd_only)
    y_ref, pd_ref = oracle.das(acq, synth.iqmod.from_storage(x.cpu()))
    assert nrmse_db(y.cpu().numpy(), y_ref) <= -100
    assert nrmse_db(pd.cpu().numpy().astype(np.float64), pd_ref) <= -100
    if dt == "c64":
        m.mach_debug_force_variant("channels_c64_cl16")
        try:
            with m.Plan(**m.plan_kwargs(acq)) as p:
                y16 = p.run(x)
                torch.cuda.synchronize()
        finally:
            m.mach_debug_force_variant(None)
        assert nrmse_db(y.cpu().numpy(), y16.cpu().numpy()) <= -115
