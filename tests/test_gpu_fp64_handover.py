"""The FP64 cell-wise tracers give the same bits whatever the number of lanes
per line, and so also when the last lines of a launch pass from the one-lane to
the sixteen-lane kernel (more than 512 line directions per SM, lanes left to the
library), which depends on the scheduling: records, step counts, counters, maps,
captured plans, step and length limits."""
import numpy as np
import pytest
import torch

from paper_1609_00724_gb300 import inputs

pytestmark = pytest.mark.gpu

FIELDS = ("q_perp", "q_foot", "q_det", "b0", "bf", "bb", "flux_f", "flux_b", "length", "lam_f", "lam_b", "x_f", "x_b",
          "steps", "face_f", "face_b", "status_f", "status_b")


@pytest.fixture(scope="module")
def qsl():
    from paper_1609_00724_gb300 import qsl as q
    q.lib()
    return q


def _field(qsl, n, mode, seed=5):
    gf = inputs.charge_field(inputs.random_charges(4, seed), n)
    return qsl.qsl_load_field(*(a.double().numpy() for a in (gf.bx, gf.by, gf.bz)), gf.xc, gf.yc, gf.zc, mode)


def _opts(qsl, lanes, tol, **kw):
    return qsl.qsl_opts_default(tol_abs=tol, tol_rel=tol, precision=qsl.QSL_FP64, integrator=qsl.QSL_DOPRI5_CELL,
                                line_lanes=lanes, **kw)


def _same(a, b):
    for k in FIELDS:
        x, y = np.ascontiguousarray(a[k]), np.ascontiguousarray(b[k])
        if x.dtype.kind == "f":
            x, y = x.view("u%d" % x.dtype.itemsize), y.view("u%d" % y.dtype.itemsize)
        assert np.array_equal(x, y), (k, int(np.sum(x != y)))


def _trace(qsl, F, seeds, o):
    rec = qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, torch.as_tensor(seeds).cuda(), o))
    st = qsl.qsl_last_stats()
    return rec, {k: st[k] for k in ("lines", "stage_evals", "accepted", "rejected", "landing")}


# the launches of 60,000 seeds hand lines over: 120,000 directions, 152 SMs
@pytest.mark.parametrize("count,mode,box,kw", [
    (1, 0, None, {}), (700, 1, None, {}), (3000, 0, "cut", {}), (60000, 0, None, {}), (60000, 1, None, {}),
    (60000, 0, "cut", {}), (60000, 1, "cut", {"max_length": 0.61}), (60000, 0, None, {"max_steps": 40})])
def test_same_bits_for_every_number_of_lanes(qsl, count, mode, box, kw):
    F = _field(qsl, 41, mode)
    seeds = inputs.random_seeds(count, 31 + count)
    seeds[::5, 2] = 0.0
    seeds[::97, 0] = 0.0  # cell faces: the plane between the two middle cells
    if box:
        lo, hi = np.array([-0.83, -1.0, 0.013]), np.array([0.91, 0.77, 0.98])
        seeds[1::2] = np.clip(seeds[1::2], lo, hi)  # some on the cut faces, some outside
        kw = dict(kw, domain_lo=lo, domain_hi=hi)
    tol = 1e-8
    a, sa = _trace(qsl, F, seeds, _opts(qsl, 1, tol, **kw))
    for lanes in (0, 3):
        b, sb = _trace(qsl, F, seeds, _opts(qsl, lanes, tol, **kw))
        _same(a, b)
        assert sa == sb
    if "max_steps" in kw:
        assert (a["status_f"] == qsl.QSL_LINE_MAXSTEPS).sum() > 100
    if "max_length" in kw:
        assert (a["status_f"] == qsl.QSL_LINE_MAXLEN).sum() > 100


def _map(m):
    return {"q": torch.empty(m * m, device="cuda"), "length": torch.empty(m * m, device="cuda"),
            "faces": torch.empty(2 * m * m, dtype=torch.uint8, device="cuda"),
            "status": torch.empty(m * m, dtype=torch.uint8, device="cuda")}


def test_maps_and_plans_repeat_bit_for_bit(qsl):
    """Two cuts of two fields, 61,250 lines in all: the maps one by one (the first
    above the rule, the second below it), and as a captured plan, replayed."""
    fields = [_field(qsl, 41, 0), _field(qsl, 33, 1, seed=9)]
    sizes = (230, 92)
    u, v = (2.0, 0.0, 0.0), (0.0, 2.0, 0.0)
    o = _opts(qsl, 0, 1e-7)
    one = [_map(m) for m in sizes]
    for F, m, out in zip(fields, sizes, one):
        qsl.qsl_q_map_2d(F, (0, 0, 0), u, v, m, m, o, **out)
    N = sum(m * m for m in sizes)
    out = {"q": torch.empty(N, device="cuda"), "length": torch.empty(N, device="cuda"),
           "faces": torch.empty(2 * N, dtype=torch.uint8, device="cuda"),
           "status": torch.empty(N, dtype=torch.uint8, device="cuda")}
    plan = qsl.Plan([(F, (0, 0, 0), u, v, m, m) for F, m in zip(fields, sizes)], o, **out)
    for _ in range(3):
        for t in out.values():
            t.fill_(7)
        plan.launch()
        torch.cuda.synchronize()
        for k in out:
            want = torch.cat([w[k] for w in one])
            assert torch.equal(out[k].view(torch.uint8), want.view(torch.uint8)), k
    again = _map(sizes[0])
    qsl.qsl_q_map_2d(fields[0], (0, 0, 0), u, v, sizes[0], sizes[0], _opts(qsl, 1, 1e-7), **again)
    for k in again:
        assert torch.equal(again[k].view(torch.uint8), one[0][k].view(torch.uint8)), k


@pytest.mark.parametrize("retrace_q,short", [(3.0, False), (200.0, True)])
@pytest.mark.parametrize("integ", [0, 2])
def test_retrace_lists_of_both_lengths(qsl, integ, retrace_q, short):
    """FP32 maps whose FP64 retrace list is above 512 line directions per SM or below
    it and not empty. Cell-wise: the same bits with one lane and with the library's
    choice. Cash-Karp: the sixteen-lane kernel agrees to FP64 rounding."""
    gf = inputs.charge_field(inputs.random_charges(4, 5), 33, dtype=torch.float32, device="cuda")
    F = qsl.qsl_load_field(gf.bx, gf.by, gf.bz, gf.xc, gf.yc, gf.zc)
    m, outs = 700, []
    for lanes in (1, 0):
        o = qsl.qsl_opts_default(integrator=integ, retrace_q=retrace_q, line_lanes=lanes)
        if integ == 2:
            o.tol_abs = o.tol_rel = 1e-6
        outs.append(_map(m))
        qsl.qsl_q_map_2d(F, (0, 0, 0), (2.0, 0.0, 0.0), (0.0, 2.0, 0.0), m, m, o, **outs[-1])
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        seeds = qsl.qsl_last_stats()["retraced"]
        assert 0 < seeds <= 256 * sms if short else seeds > 256 * sms, seeds
    for k in outs[0]:
        a, b = outs[0][k], outs[1][k]
        if integ == 2 or a.dtype == torch.uint8:
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), k
        else:
            assert torch.allclose(a, b, rtol=1e-6, atol=0, equal_nan=True), k


@pytest.mark.parametrize("n", [50, 99])
def test_lines_leave_through_every_face(qsl, n):
    """Grids whose length over their spacing rounds to more than n - 1: every line
    ends on a face within some hundred steps (one or two per cell crossed), whether
    the domain is left to the library or given as the grid's extent."""
    F = _field(qsl, n, 0)
    seeds = torch.as_tensor(inputs.random_seeds(3000, n)).cuda()
    for lanes in (1, 3):
        for kw in ({}, {"domain_lo": (-1.0, -1.0, 0.0), "domain_hi": (1.0, 1.0, 1.0)}):
            rec = qsl.lines_to_numpy(qsl.qsl_trace_seeds(F, seeds, _opts(qsl, lanes, 1e-6, max_steps=2000, **kw)))
            assert np.all(rec["status_f"] == qsl.QSL_LINE_OK) and np.all(rec["status_b"] == qsl.QSL_LINE_OK)
            assert {1, 3, 5} <= set(rec["face_f"]) | set(rec["face_b"])
