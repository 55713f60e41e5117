"""Plans and batches launched from several host threads at once: calls that share a kernel need not
share its shared-memory size."""
import threading

import numpy as np
import pytest
import torch

import synth
import paper_2604_06257_gb300 as m

pytestmark = pytest.mark.gpu


def acquisition(step, F, dt):
    """Deeper voxels per tile, hence longer windows and a larger ring, with a larger step."""
    base = synth.make_acquisition("doppler2d", "small")
    mid = len(base.elem_pos) // 2
    return base.replace(grid_dims=(64, 1, 64), grid_origin=(-32 * step, 0.0, 5e-3), grid_step=(step, 0.0, step),
                        elem_pos=base.elem_pos[mid - 16:mid + 16], n_samples=460, n_frames=F, iq_dtype=dt)


def from_two_threads(calls, n=1500):
    """Each call n times in a thread and on a stream of its own; the errors they raised."""
    errors, start = [], threading.Barrier(len(calls))

    def work(call):
        s = torch.cuda.Stream()
        start.wait()
        try:
            for i in range(n):
                call(s)
                if i % 100 == 99:
                    s.synchronize()
        except Exception as e:   # noqa: BLE001 -- reported by the test
            errors.append(e)

    ts = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    return errors


@pytest.mark.parametrize("F,dt,repack", [(32, "c64split", False), (25, "c64", True), (30, "c64", False)])
def test_two_plans_of_one_kernel(F, dt, repack):
    acqs = [acquisition(step, F, dt) for step in (1.5e-4, 2.2e-4)]
    iqs = [synth.random_iq(a.replace(iq_dtype="c64"), 7, device="cuda") for a in acqs]
    xs = [synth.iqmod.to_c64split(x) if dt == "c64split" else x for x in iqs]
    m.mach_debug_force_repack(repack)
    try:
        plans = [m.Plan(**m.plan_kwargs(a)) for a in acqs]
    finally:
        m.mach_debug_force_repack(False)
    info = [p.info() for p in plans]
    assert info[0]["variant"] == info[1]["variant"] and ("+x" in info[0]["variant"]) == repack
    if not repack:
        assert 48 << 10 < info[0]["smem_bytes"] < info[1]["smem_bytes"]
    want = [p.run(x).clone() for p, x in zip(plans, xs)]
    got = [torch.zeros_like(w) for w in want]
    torch.cuda.synchronize()
    errors = from_two_threads([lambda s, k=k: m.mach_das_run(plans[k].handle, xs[k], got[k], stream=s) for k in range(2)])
    assert not errors, errors[0]
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    for p in plans:
        p.close()


def test_two_batches():
    acqs = [acquisition(step, 25, "c64") for step in (0.8e-4, 1.2e-4)]
    xs = [synth.random_iq(a, 9, device="cuda") for a in acqs]
    ys = [torch.zeros((a.n_vox, 25), dtype=torch.complex64, device="cuda") for a in acqs]
    batches = [m.Batch([m.plan_kwargs(a)], shapes=[(2, 8, None)]) for a in acqs]
    for b, x, y in zip(batches, xs, ys):
        b.bind([x], [y], None)
        b.run()
    torch.cuda.synchronize()
    want = [y.clone() for y in ys]
    errors = from_two_threads([lambda s, b=b: b.run(stream=s) for b in batches])
    assert not errors, errors[0]
    for a, b in zip(ys, want):
        assert torch.equal(a, b)
    for b in batches:
        b.close()
