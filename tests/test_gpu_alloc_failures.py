"""Device allocations that fail one after another while repacking plans and batches are made and
run: each call either reports OUT OF MEMORY, or does without the workspace and beamforms by
the kernel that reads the ensemble directly; nothing is left behind."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_06257_gb300 as m
from metrics import nrmse_db
from test_gpu_repack import dense, repack_small_grids, stored   # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def failing(n, make):
    """make() with the n-th allocation failing; (result or None, whether the failure was reached)."""
    m.mach_debug_fail_alloc_after(n)
    try:
        got = make()
    except m.MachError as e:
        assert e.status == m.MACH_ERR_OOM
        return None, True
    finally:
        left = m.mach_debug_allocs_to_failure()
        m.mach_debug_fail_alloc_after(0)
    return got, left == 0


def direct(acq, x, name):
    m.mach_debug_force_variant(name)
    try:
        with m.Plan(**m.plan_kwargs(acq)) as p:
            return p.power_doppler(x, want_y=True)
    finally:
        m.mach_debug_force_variant(None)


@pytest.mark.parametrize("F,dt", [(25, "c64"), (40, "f16x2")])
def test_plans_do_without_the_workspace(F, dt):
    acq = dense(F, dt, 2, 3)
    x, _ = stored(acq, F)
    kw = m.plan_kwargs(acq)
    with m.Plan(**kw) as p:
        name = p.info()["variant"]
        base = p.info()["device_bytes"]
    assert "+x" in name
    pd_d, y_d = direct(acq, x, name.split("+")[0])
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    without, n, reached = 0, 0, True
    while reached:
        n += 1
        plan, reached = failing(n, lambda: m.Plan(**kw))
        if plan is None:
            continue
        with plan as p:
            if reached:      # the plan did without what failed
                without += 1
                assert p.info()["variant"] == name.split("+")[0] and p.info()["device_bytes"] < base
                pd, y = p.power_doppler(x, want_y=True)
                torch.cuda.synchronize()
                assert torch.equal(y, y_d) and torch.equal(pd, pd_d)
    assert without >= 4 and n > without
    torch.cuda.synchronize()
    assert abs(torch.cuda.mem_get_info()[0] - free0) < (64 << 20)


def test_a_run_without_memory_takes_the_direct_kernel():
    acq = dense(25, "c64", 2, 3)
    x, _ = stored(acq, 1)
    with m.Plan(**m.plan_kwargs(acq)) as p:
        name = p.info()["variant"]
        pd_d, y_d = direct(acq, x, name.split("+")[0])
        (pd, y), reached = failing(1, lambda: p.power_doppler(x, want_y=True))
        assert reached
        torch.cuda.synchronize()
        assert torch.equal(y, y_d) and torch.equal(pd, pd_d)
        pd, y = p.power_doppler(x, want_y=True)          # the next run has its workspace again
        torch.cuda.synchronize()
        assert not torch.equal(y, y_d) and nrmse_db(y.cpu().numpy(), y_d.cpu().numpy()) <= -110


def test_batches_do_without_the_workspace():
    acqs = [dense(F, "c64", 2 + i % 2, 1 + i % 3) for i, F in enumerate([2, 5, 16, 25, 41])]
    xs = [stored(a, i)[0] for i, a in enumerate(acqs)]
    kws = [m.plan_kwargs(a) for a in acqs]

    def run(b):
        ys = [torch.zeros((a.n_vox, a.n_frames), dtype=torch.complex64, device="cuda") for a in acqs]
        b.bind(xs, ys, None)
        b.run()
        torch.cuda.synchronize()
        return ys

    with m.Batch(kws) as b:
        info, want = b.info(), run(b)
    with m.Batch(kws, shapes=[(s[0], s[1], None) for s in info["shapes"]]) as b:
        lanes, y_lanes = b.info()["items"], run(b)
    assert lanes != info["items"]
    for a, x, y in zip(acqs, xs, want):
        idx = np.arange(0, a.n_vox, 17)
        assert nrmse_db(y.cpu().numpy()[idx], oracle.das(a, x.cpu(), idx)[0]) <= -100
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    without, partly, n, reached = 0, 0, 0, True
    while reached:
        n += 1
        batch, reached = failing(n, lambda: m.Batch(kws))
        if batch is None:
            continue
        with batch as b:
            if not reached:
                assert all(torch.equal(y, w) for y, w in zip(run(b), want))
                continue
            for y, w, l in zip(run(b), want, y_lanes):
                assert torch.equal(y, w) or torch.equal(y, l)
            if b.info()["items"] == lanes:
                without += 1
            else:
                partly += 1       # one instance's own tables failed: that one on its lanes
    # the workspace and each of the tile shapes' item lists
    assert without >= 4 and partly >= 3, (without, partly)
    torch.cuda.synchronize()
    assert abs(torch.cuda.mem_get_info()[0] - free0) < (64 << 20)


def run_concurrently(plans, acqs):
    """Runs of two plans at once have a workspace each, also while a third plan goes."""
    xs = [stored(a, i)[0] for i, a in enumerate(acqs[:2])]
    want = [p.run(x).clone() for p, x in zip(plans[::2], xs)]
    got = [torch.zeros_like(w) for w in want]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    for _ in range(3):
        for p, x, y, s in zip(plans[::2], xs, got, streams):
            m.mach_das_run(p.handle, x, y, stream=s)
    plans.pop().close()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_idle_plans_share_one_workspace():
    """Device memory that plans hold between runs: one workspace for all of them, none after the last."""
    acqs = [dense(F, "c64split", 2, 3) for F in (2048, 2028, 2016)]
    ws = 3 * 24 * 200 * 8 * 2048

    def held():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return free0 - torch.cuda.mem_get_info()[0]

    free0 = 0
    warm = [m.Plan(**m.plan_kwargs(a)) for a in acqs for _ in range(2)]   # modules load, torch's own blocks come
    run_concurrently(warm, acqs)
    for p in warm:
        p.close()
    free0 = -held()
    plans = [m.Plan(**m.plan_kwargs(a)) for a in acqs for _ in range(2)]
    try:
        assert all("+x" in p.info()["variant"] and p.info()["device_bytes"] > 0.95 * ws for p in plans)
        assert held() < 2 * ws
        run_concurrently(plans, acqs)
        assert held() < 2 * ws
    finally:
        for p in plans:
            p.close()
    assert held() < (64 << 20)
