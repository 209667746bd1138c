"""What a launch reports and does when the library chooses for the caller: the
refill threshold (automatic, 1, 4, 8: the same bits), the resident blocks that a
caller allows, the watchdog's one clock per launch."""
import numpy as np
import pytest
import torch

from paper_1609_00724_gb300 import inputs

pytestmark = pytest.mark.gpu

U, V = (2.0, 0.0, 0.0), (0.0, 2.0, 0.0)


@pytest.fixture(scope="module")
def qsl():
    from paper_1609_00724_gb300 import qsl as q
    q.lib()
    return q


def _field(qsl, n, seed=5, mode=0):
    gf = inputs.charge_field(inputs.random_charges(4, seed), n, dtype=torch.float32, device="cuda")
    return qsl.qsl_load_field(gf.bx, gf.by, gf.bz, gf.xc, gf.yc, gf.zc, mode)


def _map(qsl, F, m, o):
    out = {"q": torch.empty(m * m, device="cuda"), "length": torch.empty(m * m, device="cuda"),
           "faces": torch.empty(2 * m * m, dtype=torch.uint8, device="cuda"),
           "status": torch.empty(m * m, dtype=torch.uint8, device="cuda")}
    qsl.qsl_q_map_2d(F, (0, 0, 0), U, V, m, m, o, **out)
    return out, qsl.qsl_last_stats()


def test_handed_over_lines_keep_the_launch_clock(qsl):
    """An FP64 cell-wise launch of 120,000 directions runs in two kernels of
    comparable length (the second takes up the lines that the first hands over):
    a watchdog of 40 to 80 percent of their time together stops it, whichever of
    the two is running then."""
    F = _field(qsl, 65, mode=1)
    seeds = torch.as_tensor(inputs.random_seeds(60000, 43)).cuda()
    o = qsl.qsl_opts_default(tol_abs=1e-11, tol_rel=1e-11, integrator=qsl.QSL_DOPRI5_CELL, precision=qsl.QSL_FP64)
    for _ in range(2):
        rec = qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, seeds, o))
        ms = qsl.qsl_last_stats()["kernel_ms"]
    for part in (0.4, 0.5, 0.6, 0.7, 0.8):
        o.timeout_s = part * ms * 1e-3
        cut = qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, seeds, o))
        with pytest.raises(qsl.QslError) as e:
            qsl.qsl_last_stats()
        assert e.value.code == qsl.QSL_ETIMEOUT, part
        late = (cut["status_f"] == qsl.QSL_LINE_TIMEOUT) | (cut["status_b"] == qsl.QSL_LINE_TIMEOUT)
        assert late.any() and not late.all()
        for k in ("q_perp", "length", "steps"):
            assert np.array_equal(cut[k][~late], rec[k][~late], equal_nan=k != "steps"), k


@pytest.mark.parametrize("integ,count", [(2, 4000), (0, 4000)])
def test_watchdog_and_step_limit_with_sixteen_lanes(qsl, integ, count):
    """Few lines in FP64 run on sixteen lanes each with either stepper: one
    microsecond stops them after the next check (every 64 loop iterations), a step
    limit at that many steps, and the next call runs to completion."""
    F = _field(qsl, 65)
    seeds = torch.as_tensor(inputs.random_seeds(count, 43)).cuda()
    kw = dict(tol_abs=1e-9, tol_rel=1e-9, integrator=integ, precision=qsl.QSL_FP64)
    rec = qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, seeds, qsl.qsl_opts_default(**kw)))
    qsl.qsl_last_stats()
    cut = qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, seeds, qsl.qsl_opts_default(timeout_s=1e-6, **kw)))
    with pytest.raises(qsl.QslError) as e:
        qsl.qsl_last_stats()
    assert e.value.code == qsl.QSL_ETIMEOUT
    st = np.concatenate([cut["status_f"], cut["status_b"]])
    assert np.sum(st == qsl.QSL_LINE_TIMEOUT) > 100
    assert np.all((st == qsl.QSL_LINE_TIMEOUT) | (st == qsl.QSL_LINE_OK))
    few = qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, seeds, qsl.qsl_opts_default(max_steps=30, **kw)))
    qsl.qsl_last_stats()
    st = np.concatenate([few["status_f"], few["status_b"]])
    assert np.sum(st == qsl.QSL_LINE_MAXSTEPS) > 100
    both = (few["status_f"] == qsl.QSL_LINE_MAXSTEPS) & (few["status_b"] == qsl.QSL_LINE_MAXSTEPS)
    assert both.any() and np.all(few["steps"][both] == 60)
    full = (few["status_f"] == qsl.QSL_LINE_OK) & (few["status_b"] == qsl.QSL_LINE_OK)
    assert np.array_equal(few["steps"][full], rec["steps"][full])


@pytest.mark.parametrize("kw", [dict(integrator=2, tol_abs=1e-5, tol_rel=1e-5), dict(tol_abs=1e-2, tol_rel=1e-2)])
def test_refill_threshold_is_reported_as_used(qsl, kw):
    """900 x 900 seeds are far more than four times the resident lanes (at most 64
    warps per SM), 60 x 60 far fewer. A line's result does not depend on when its
    lane took it up: every threshold gives the same bits."""
    F = _field(qsl, 33)
    outs, used = [], []
    for refill in (0, 1, 4, 8):
        out, st = _map(qsl, F, 900, qsl.qsl_opts_default(refill_min=refill, retrace_q=0.0, **kw))
        outs.append(out)
        used.append(st["refill_min"])
    assert used == [8, 1, 4, 8]
    for out in outs[1:]:
        for k in out:
            assert torch.equal(out[k].view(torch.uint8), outs[0][k].view(torch.uint8)), k
    o = qsl.qsl_opts_default(**kw)
    _, st = _map(qsl, F, 60, o)
    assert st["refill_min"] == 1
    q = torch.empty(3600, device="cuda")
    plan = qsl.Plan([(F, (0, 0, 0), U, V, 60, 60)], o, q=q, length=torch.empty_like(q),
                    faces=torch.empty(7200, dtype=torch.uint8, device="cuda"),
                    status=torch.empty(3600, dtype=torch.uint8, device="cuda"))
    plan.launch()
    assert plan.stats()["refill_min"] == 1


@pytest.mark.parametrize("integ", [0, 2])
def test_allowed_blocks_bound_the_sixteen_lane_kernels(qsl, integ):
    """One resident block of one warp per SM against as many as fit: FP64 warp
    instructions take 64 cycles of a warp and 19 of an SM, so four warps per SM and
    more are at least twice as fast as one."""
    F = _field(qsl, 65)
    seeds = torch.as_tensor(inputs.random_seeds(4000, 43)).cuda()
    ms = []
    for blocks in (1, 0):
        o = qsl.qsl_opts_default(tol_abs=1e-6, tol_rel=1e-6, integrator=integ, precision=qsl.QSL_FP64, warps_per_block=1,
                                 blocks_per_sm=blocks)
        best = np.inf
        for _ in range(4):
            qsl.qsl_trace_seeds(F, seeds, o)
            best = min(best, qsl.qsl_last_stats()["kernel_ms"])
        ms.append(best)
    assert ms[0] > 1.6 * ms[1], ms


@pytest.mark.parametrize("order", [2, 3])
def test_refill_rule_of_the_higher_orders(qsl, order):
    """Cash-Karp with the deviations in FP32: no wait on a small field, where the
    idle lanes cost more than the refills, 8 lanes on one that outgrows the caches."""
    used = []
    for n in (33, 120):
        F, outs = _field(qsl, n), []
        for refill in (0, 1, 8):
            out, st = _map(qsl, F, 320, qsl.qsl_opts_default(refill_min=refill, retrace_q=0.0, interp_order=order))
            outs.append(out)
            used.append(st["refill_min"])
        for k in outs[0]:
            assert all(torch.equal(o[k].view(torch.uint8), outs[0][k].view(torch.uint8)) for o in outs[1:]), k
    assert used == [1, 1, 8, 8, 1, 8]


def test_raw_cash_karp_maps_of_many_lines_take_one_lane(qsl):
    """FP64 Cash-Karp on a raw field at a loose tolerance: 30,000 seeds (above 352
    line directions per SM) run on one lane each, with the bits of line_lanes = 1;
    20,000, and 30,000 at a tight tolerance, on sixteen (rounding apart; how far is
    the lane tests' question)."""
    F = _field(qsl, 33, mode=1)
    for count, tol, same in ((30000, 1e-2, True), (20000, 1e-2, False), (30000, 1e-4, False)):
        seeds = torch.as_tensor(inputs.random_seeds(count, 7)).cuda()
        a, b = [qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, seeds, qsl.qsl_opts_default(
            tol_abs=tol, tol_rel=tol, precision=qsl.QSL_FP64, line_lanes=lanes))) for lanes in (1, 0)]
        assert np.array_equal(a["face_f"], b["face_f"]) and np.array_equal(a["status_b"], b["status_b"])
        assert np.array_equal(a["q_perp"], b["q_perp"], equal_nan=True) == same, count
