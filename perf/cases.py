"""Performance cases: the work a user of this package has it do, through the
public binding (paper_1609_00724_gb300.qsl) and the learned-proposal helpers
(paper_1609_00724_gb300.learned).

A case is a dict of plain values with a "kind"; listed() names the fixed ones,
draw(rng) gives one more of the same ranges. prepare() builds the inputs and
the handles a program keeps (packed fields, captured plans, networks, sample
buffers), run() is one pass through the entry points.

Fields are the package's synthetic ones: potential fields of point charges
below the lower boundary (Cartesian box or spherical wedge) and the linear
hyperbolic field, whose squashing factor has a closed form. The charges, the
field constants and the network's data come from the seed, the sizes from the
case.
"""
import math

import numpy as np
import torch

from paper_1609_00724_gb300 import inputs, learned, qsl

DEV = "cuda"
BOX_U, BOX_V = (2.0, 0.0, 0.0), (0.0, 2.0, 0.0)  # the whole z = 0 plane of the box

# Mean tracer work of one seed (both directions) per 256 grid cells along an
# axis, from the counters of a 1024^2 map of a 4-charge field on 256^3: 806
# right-hand-side evaluations of the cell-wise stepper at 227 FLOP each. Lines
# of a coarser grid cross proportionally fewer cells. The Cash-Karp stepper at
# tight tolerances is counted with the same necessary work.
STAGES_PER_SEED_256, FLOP_PER_STAGE = 806.0, 227.0


def listed():
    return [
        # A user looks at a few field lines: host seeds in, host records out, the smallest call there is.
        {"name": "seeds_host_48", "kind": "seeds", "n": 64, "charges": 4, "seeds": 48, "host": True, "integ": "cell",
         "tol": 1e-6},
        # The validation map of the README's linear field, raw interpolation, footpoint Q against its closed form.
        {"name": "hyperbolic_256", "kind": "hyper", "n": 64, "m": 256},
        # What a first-time user gets: default options (Cash-Karp, tolerance 1e-2) on an ordinary slice.
        {"name": "map_default_512", "kind": "map", "n": 128, "charges": 4, "nu": 512, "nv": 512, "integ": "ck",
         "tol": 1e-2, "hmax": 2.0, "fp64": False, "order": 1, "raw": False},
        # The photospheric Q map of the benchmark's field at the settings its tuner picks.
        {"name": "map_cell_1024", "kind": "map", "n": 256, "charges": 4, "nu": 1024, "nv": 1024, "integ": "cell",
         "tol": 1e-5, "hmax": 4.0, "fp64": False, "order": 1, "raw": False},
        # The same path in FP64 everywhere, used to check a map; odd sizes.
        {"name": "map_fp64_321", "kind": "map", "n": 128, "charges": 4, "nu": 321, "nv": 257, "integ": "cell",
         "tol": 1e-7, "hmax": 2.0, "fp64": True, "order": 1, "raw": False},
        # A spherical slice at the lower radius (longitude x latitude), Cash-Karp at a tight tolerance.
        {"name": "map_spherical_512", "kind": "sphere", "np": 256, "nt": 192, "nr": 128, "charges": 6, "nu": 512,
         "nv": 384, "tol": 1e-7},
        # A Q/FLL volume and its 3D FLEDGE map: many long lines, the largest launch.
        {"name": "volume_256", "kind": "volume", "n": 256, "charges": 8, "nx": 256, "ny": 256, "nz": 128,
         "tol": 1e-7},
        # Many cuts of many fields of different sizes replayed as one captured plan.
        {"name": "plan_16_fields", "kind": "plan", "fields": 16, "sizes": 4, "n_lo": 64, "n_hi": 256, "m_lo": 256,
         "m_hi": 1024, "tol": 1e-7},
        # The headline workload: field load, coarse map, FLL-jump refinement, both grids, FLEDGE of the length grid.
        {"name": "refine_1024_4096", "kind": "refine2", "n": 256, "charges": 4, "coarse": 1024, "levels": 2,
         "tau": 0.05, "tol": 1e-5, "hmax": 4.0},
        # One training volume of the learned proposal: a 3D refinement of two orders, grids one order coarser.
        {"name": "refine_volume_64", "kind": "refine3", "n": 128, "charges": 8, "cx": 64, "cy": 64, "cz": 32,
         "levels": 2, "tau": 0.05, "tol": 1e-6, "iters": 64, "proposal": False},
        # Where to refine a large coarse volume: features and network over all its slices.
        {"name": "propose_128x256x256", "kind": "infer", "nz": 128, "ny": 256, "nx": 256},
        # One optimiser step of the network at the size it is trained with.
        {"name": "train_32x64x64", "kind": "train", "batch": 32, "h": 64, "w": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["seeds", "hyper", "map", "map", "sphere", "volume", "plan", "refine2", "refine3", "infer",
                       "train"])
    if kind == "seeds":
        return {"kind": kind, "n": _log_int(rng, 33, 192), "charges": rng.randint(2, 8),
                "seeds": _log_int(rng, 1, 20000), "host": rng.random() < 0.5, "integ": rng.choice(["cell", "ck"]),
                "tol": rng.choice([1e-2, 1e-5, 1e-6])}
    if kind == "hyper":
        return {"kind": kind, "n": _log_int(rng, 24, 128), "m": _log_int(rng, 31, 400)}
    if kind == "map":
        fp64 = rng.random() < 0.2
        integ = rng.choice(["cell", "cell", "ck"])
        order = 3 if integ == "ck" and not fp64 and rng.random() < 0.25 else 1
        return {"kind": kind, "n": _log_int(rng, 48, 128 if fp64 else 256), "charges": rng.randint(3, 8),
                "nu": _log_int(rng, 40, 256 if fp64 else 1024), "nv": _log_int(rng, 40, 256 if fp64 else 768),
                "integ": integ, "tol": rng.choice([1e-5, 1e-6]) if integ == "cell" else rng.choice([1e-2, 1e-5]),
                "hmax": rng.choice([2.0, 4.0]), "fp64": fp64, "order": order, "raw": rng.random() < 0.25}
    if kind == "sphere":
        return {"kind": kind, "np": _log_int(rng, 48, 256), "nt": _log_int(rng, 40, 192),
                "nr": _log_int(rng, 32, 128), "charges": rng.randint(3, 8), "nu": _log_int(rng, 40, 512),
                "nv": _log_int(rng, 40, 384), "tol": rng.choice([1e-4, 1e-6])}
    if kind == "volume":
        return {"kind": kind, "n": _log_int(rng, 64, 224), "charges": rng.randint(3, 8),
                "nx": _log_int(rng, 32, 224), "ny": _log_int(rng, 32, 224), "nz": _log_int(rng, 17, 112),
                "tol": rng.choice([1e-5, 1e-6, 1e-7])}
    if kind == "plan":
        return {"kind": kind, "fields": rng.randint(2, 12), "sizes": rng.randint(0, 1 << 20), "n_lo": 48,
                "n_hi": rng.randint(96, 224), "m_lo": 64, "m_hi": rng.randint(256, 896),
                "tol": rng.choice([1e-5, 1e-6])}
    if kind == "refine2":
        return {"kind": kind, "n": _log_int(rng, 64, 256), "charges": rng.randint(3, 8),
                "coarse": 1 << rng.randint(6, 10), "levels": rng.randint(1, 2), "tau": rng.choice([0.03, 0.05, 0.1]),
                "tol": rng.choice([1e-5, 1e-6]), "hmax": rng.choice([2.0, 4.0])}
    if kind == "refine3":
        c = 1 << rng.randint(4, 6)
        return {"kind": kind, "n": _log_int(rng, 48, 128), "charges": rng.randint(4, 12), "cx": c, "cy": c,
                "cz": c // 2, "levels": rng.randint(1, 2), "tau": 0.05, "tol": 1e-6,
                "iters": rng.choice([2, 64]), "proposal": rng.random() < 0.5}
    if kind == "infer":
        return {"kind": kind, "nz": _log_int(rng, 1, 96), "ny": _log_int(rng, 24, 256), "nx": _log_int(rng, 24, 256)}
    return {"kind": "train", "batch": _log_int(rng, 2, 48), "h": _log_int(rng, 24, 128), "w": _log_int(rng, 24, 128)}


# ---------------------------------------------------------------- inputs
def _load(gf, raw=False):
    return qsl.qsl_load_field(gf.bx, gf.by, gf.bz, gf.xc, gf.yc, gf.zc,
                              qsl.QSL_RAW_B if raw else qsl.QSL_PAPER_NORMALIZE_FIRST)


def _charge_field(n, charges, seed):
    return inputs.charge_field(inputs.random_charges(charges, seed), n, dtype=torch.float32, device=DEV, slab=64)


def _opts(integ, tol, hmax=2.0, **kw):
    return qsl.qsl_opts_default(integrator=qsl.QSL_DOPRI5_CELL if integ == "cell" else qsl.QSL_RKCK54, tol_abs=tol,
                                tol_rel=tol, h_max=hmax, **kw)


def _map_out(N):
    return {"q": torch.empty(N, device=DEV), "length": torch.empty(N, device=DEV),
            "faces": torch.empty(2 * N, dtype=torch.uint8, device=DEV),
            "status": torch.empty(N, dtype=torch.uint8, device=DEV)}


def _hyper_constants(seed):
    rng = np.random.default_rng([seed, 1])
    return float(rng.uniform(2.0, 3.5)), float(rng.uniform(0.8, 1.25))


def _plan_sizes(case):
    rng = np.random.default_rng([case["sizes"], 2])
    return [(int(rng.integers(case["n_lo"], case["n_hi"] + 1)), int(rng.integers(case["m_lo"], case["m_hi"] + 1)))
            for _ in range(case["fields"])]


def _generator(seed, salt):
    return torch.Generator(device=DEV).manual_seed(seed * 16 + salt)


def _coarse_volume(case, seed):
    """Lengths and Q of a coarse volume: smooth lobes of field-line length that
    jump across a few curved surfaces, Q log-normal and raised near the jumps,
    a few pixels without a Q."""
    g = _generator(seed, 3)
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    z = torch.linspace(0, 1, nz, device=DEV).view(-1, 1, 1)
    y = torch.linspace(-1, 1, ny, device=DEV).view(1, -1, 1)
    x = torch.linspace(-1, 1, nx, device=DEV).view(1, 1, -1)
    c = torch.rand(5, 4, generator=g, device=DEV) * 2 - 1
    L = torch.full((nz, ny, nx), 1.5, device=DEV)
    near = torch.zeros_like(L)
    for k in range(5):
        s = x * (1 + c[k, 0]) + y * c[k, 1] * 2 + z * c[k, 2] + 0.4 * torch.sin(3 * x * y + 4 * c[k, 3]) + 0.3 * c[k, 2]
        L = L + 0.2 * torch.tanh(s) + 0.25 * (s > 0)
        near = torch.maximum(near, torch.exp(-(s * 40) ** 2))
    noise = torch.randn((nz, ny, nx), generator=g, device=DEV)
    Q = 2 + 10 ** (0.3 + 0.25 * noise + 4 * near)
    Q[torch.rand((nz, ny, nx), generator=g, device=DEV) < 1e-3] = float("nan")
    return L.contiguous(), Q.contiguous()


def _features64(L, Q):
    """FLEDGE of the length volume and the two network channels, in 64 bits."""
    L, Q = L.double(), Q.double()
    P = L[None, None]
    for d in (2, 3, 4):  # half-sample-symmetric boundary
        P = torch.cat([P.narrow(d, 0, 1), P, P.narrow(d, P.shape[d] - 1, 1)], d)
    P = P[0, 0]
    g2 = torch.zeros_like(L)
    for axis in range(3):
        t = P
        for d in range(3):
            n = t.shape[d] - 2
            lo, mid, hi = t.narrow(d, 0, n), t.narrow(d, 1, n), t.narrow(d, 2, n)
            t = hi - lo if d == axis else lo + 2 * mid + hi
        g2 += t * t
    S = torch.sqrt(g2)
    smax = torch.clamp(S.flatten(1).max(1).values, min=1e-12).view(-1, 1, 1)
    q = torch.where(torch.isnan(Q), torch.full_like(Q, 2.0), Q)
    x1 = torch.clamp((torch.log10(torch.clamp(q, min=2.0)) - 2) * 0.5, -2.0, 3.0)
    return torch.stack([S / smax, x1], 1)


def _params(seed):
    """Network weights as training starts from them, with small biases."""
    p = learned.init_params(seed % 100003)
    rng = np.random.default_rng([seed, 4])
    for o, n in ((576, 32), (576 + 32 + 9216, 32), (qsl.QSL_CNN_NPARAMS - 1, 1)):
        p[o:o + n] = rng.uniform(-0.1, 0.1, n)
    return p


def _batch(case, seed):
    """Training inputs, labels (cells near the length jumps, some missing) and
    the positive-class weight."""
    b, h, w = case["batch"], case["h"], case["w"]
    X = _features64(*_coarse_volume({"nz": b, "ny": h, "nx": w}, seed)).float().contiguous()
    keep = torch.rand((b, h, w), generator=_generator(seed, 6), device=DEV) < 0.9
    return X, ((X[:, 0] > 0.3) & keep).float().contiguous(), 4.0 + seed % 8


def _mask(case, seed):
    """Proposal mask of a coarse volume: blobs over a few percent of the cells."""
    g = _generator(seed, 5)
    shape = (case["cz"], case["cy"], case["cx"])
    r = torch.rand((1, 1) + tuple(max(2, s // 4) for s in shape), generator=g, device=DEV)
    r = torch.nn.functional.interpolate(r, size=shape, mode="trilinear", align_corners=True)[0, 0]
    return (r > 0.85).to(torch.uint8).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "seeds":
        F = _load(_charge_field(case["n"], case["charges"], seed))
        s = inputs.random_seeds(case["seeds"], seed + 1, margin=0.02)
        return {"case": case, "F": F, "seeds": s if case["host"] else torch.as_tensor(s).cuda(),
                "o": _opts(case["integ"], case["tol"])}
    if kind == "hyper":
        lam, b0 = _hyper_constants(seed)
        gf = inputs.hyperbolic_field(case["n"], lam, b0)
        t = [torch.as_tensor(a).cuda() for a in (gf.bx, gf.by, gf.bz)]
        F = qsl.qsl_load_field(*t, gf.xc, gf.yc, gf.zc, qsl.QSL_RAW_B)
        return {"case": case, "F": F, "o": _opts("cell", 1e-7, q_form=qsl.QSL_Q_FOOT), "out": _map_out(case["m"] ** 2)}
    if kind == "map":
        F = _load(_charge_field(case["n"], case["charges"], seed), case["raw"])
        o = _opts(case["integ"], case["tol"], case["hmax"], interp_order=case["order"],
                  precision=qsl.QSL_FP64 if case["fp64"] else qsl.QSL_FP32_MIXED)
        return {"case": case, "F": F, "o": o, "out": _map_out(case["nu"] * case["nv"])}
    if kind == "sphere":
        gf = inputs.spherical_charge_field(inputs.random_wedge_charges(case["charges"], seed),
                                           (case["np"], case["nt"], case["nr"]), dtype=torch.float32, device=DEV,
                                           slab=64)
        F = qsl.qsl_set_geometry(_load(gf), qsl.QSL_GEOM_SPHERICAL)
        return {"case": case, "F": F, "o": _opts("ck", case["tol"]), "out": _map_out(case["nu"] * case["nv"])}
    if kind == "volume":
        F = _load(_charge_field(case["n"], case["charges"], seed))
        shape = (case["nz"], case["ny"], case["nx"])
        return {"case": case, "F": F, "o": _opts("cell", case["tol"]), "out": _map_out(math.prod(shape)),
                "S": torch.empty(shape, device=DEV)}
    if kind == "plan":
        items = []
        for k, (n, m) in enumerate(_plan_sizes(case)):
            items.append((_load(_charge_field(n, 4, seed * 64 + k)), (0, 0, 0), BOX_U, BOX_V, m, m))
        out = _map_out(sum(it[4] * it[5] for it in items))
        return {"case": case, "plan": qsl.Plan(items, _opts("cell", case["tol"]), **out), "out": out}
    if kind == "refine2":
        eff = case["coarse"] << case["levels"]
        smp = learned.Samples(eff * eff)
        return {"case": case, "gf": _charge_field(case["n"], case["charges"], seed), "smp": smp,
                "o": _opts("cell", case["tol"], case["hmax"]),
                "spec": learned.plane_spec(case["coarse"], case["levels"], case["tau"]),
                "qg": torch.empty((eff, eff), device=DEV), "lg": torch.empty((eff, eff), device=DEV),
                "S": torch.empty((eff, eff), device=DEV)}
    if kind == "refine3":
        cs, lev = (case["cx"], case["cy"], case["cz"]), case["levels"]
        smp = learned.Samples(math.prod(cs) << (3 * lev))
        mask = _mask(case, seed) if case["proposal"] else None
        mask_d = torch.empty_like(mask) if mask is not None else None
        spec = learned.volume_spec(cs, lev, case["tau"], max_iters=case["iters"], proposal=mask_d)
        spec.out_order = spec.max_order - 1
        shape = tuple((c << lev) >> 1 for c in cs[::-1])
        return {"case": case, "F": _load(_charge_field(case["n"], case["charges"], seed)), "smp": smp,
                "o": _opts("cell", case["tol"]), "spec": spec, "mask": mask, "mask_d": mask_d,
                "qg": torch.empty(shape, device=DEV), "lg": torch.empty(shape, device=DEV)}
    if kind == "infer":
        L, Q = _coarse_volume(case, seed)
        return {"case": case, "L": L, "Q": Q, "net": qsl.Cnn(_params(seed))}
    X, Y, pos = _batch(case, seed)
    return {"case": case, "net": qsl.Cnn(_params(seed)), "X": X, "Y": Y, "pos": pos,
            "loss": torch.zeros(1, device=DEV), "grad": torch.zeros(qsl.QSL_CNN_NPARAMS, device=DEV)}


# ---------------------------------------------------------------- one pass
def _records(r):
    """Typed views of the qsl_line records (no copies)."""
    if isinstance(r, np.ndarray):
        return {k: r[k] for k in qsl.QSL_LINE_DTYPE.names if k != "pad0"}
    f4 = r.view(torch.float32).view(-1, 28)
    return {"f8": r.view(torch.float64).view(-1, 14)[:, :8], "len": f4[:, 16:19], "ends": f4[:, 20:26],
            "steps": r.view(torch.int32).view(-1, 28)[:, 26], "bytes": r.view(-1, 112)[:, 108:112]}


def _refined(s, n, grids):
    """The sample arrays at their full capacity, rows past the n samples cleared (they hold scratch), and the grids."""
    smp = s["smp"]
    for a in (smp.key[n:], smp.q[n:], smp.L[n:], smp.faces[2 * n:], smp.status[n:]):
        a.zero_()
    return {"n": n, "key": smp.key, "q": smp.q, "length": smp.L, "faces": smp.faces, "status": smp.status,
            **{k: s[k] for k in grids}}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "seeds":
        return _records(qsl.qsl_trace_seeds(s["F"], s["seeds"], s["o"]))
    if kind == "hyper":
        qsl.qsl_q_map_2d(s["F"], (0, 0, 0), BOX_U, BOX_V, case["m"], case["m"], s["o"], **s["out"])
        return s["out"]
    if kind == "map":
        qsl.qsl_q_map_2d(s["F"], (0, 0, 0), BOX_U, BOX_V, case["nu"], case["nv"], s["o"], **s["out"])
        return s["out"]
    if kind == "sphere":
        (p0, p1), (t0, t1), (r0, _) = inputs.WEDGE
        qsl.qsl_q_map_2d(s["F"], (0.5 * (p0 + p1), 0.5 * (t0 + t1), r0), (p1 - p0, 0, 0), (0, t1 - t0, 0), case["nu"],
                         case["nv"], s["o"], **s["out"])
        return s["out"]
    if kind == "volume":
        lo, hi = [b[0] for b in inputs.BOX], [b[1] for b in inputs.BOX]
        qsl.qsl_q_volume_3d(s["F"], lo, hi, case["nx"], case["ny"], case["nz"], s["o"], **s["out"])
        qsl.qsl_fledge(s["out"]["length"].view(s["S"].shape), s["S"])
        return {**s["out"], "S": s["S"]}
    if kind == "plan":
        s["plan"].launch()
        return s["out"]
    if kind == "refine2":
        F = _load(s["gf"])
        smp = s["smp"]
        n, _, _, _ = qsl.qsl_refine(F, s["spec"], s["o"], smp.key, smp.q, smp.L, smp.faces, smp.status, 0, s["qg"],
                                    s["lg"])
        qsl.qsl_fledge(s["lg"], s["S"])
        return _refined(s, n, ("qg", "lg", "S"))
    if kind == "refine3":
        if s["mask"] is not None:
            qsl.qsl_mask_dilate(s["mask"], s["mask_d"])
        smp = s["smp"]
        n, _, _, _ = qsl.qsl_refine(s["F"], s["spec"], s["o"], smp.key, smp.q, smp.L, smp.faces, smp.status, 0,
                                    s["qg"], s["lg"])
        return _refined(s, n, ("qg", "lg"))
    if kind == "infer":
        X = learned.features_slices(s["L"], s["Q"])
        return {"X": X, "prob": learned.predict(s["net"], X)}
    s["net"].loss_grad(s["X"], s["Y"], s["pos"], s["loss"], s["grad"])
    s["net"].adam(s["grad"], lr=2e-3)
    return {"loss": s["loss"], "grad": s["grad"]}


# ---------------------------------------------------------------- necessary work
def _trace_work(seeds, n, vertices, out_bytes=11):
    return {"bytes": 16.0 * vertices + out_bytes * seeds,
            "flops": seeds * STAGES_PER_SEED_256 * (n / 256.0) * FLOP_PER_STAGE}


def work(case):
    kind = case["kind"]
    if kind == "seeds":
        return _trace_work(case["seeds"], case["n"], 0, 24 + 112 + 128 * case["n"])
    if kind == "hyper":
        return _trace_work(case["m"] ** 2, 0.4 * case["n"], case["n"] ** 3)
    if kind == "map":
        return _trace_work(case["nu"] * case["nv"], case["n"], case["n"] ** 3)
    if kind == "sphere":
        return _trace_work(case["nu"] * case["nv"], case["np"], case["np"] * case["nt"] * case["nr"])
    if kind == "volume":
        return _trace_work(case["nx"] * case["ny"] * case["nz"], case["n"], case["n"] ** 3, 15)
    if kind == "plan":
        parts = [_trace_work(m * m, n, n ** 3) for n, m in _plan_sizes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "refine2":
        # the coarse map, about 6 % more refined samples, the field read and both grids and FLEDGE written
        cells = float(case["coarse"] << case["levels"]) ** 2
        w = _trace_work(1.06 * case["coarse"] ** 2, case["n"], case["n"] ** 3, 19)
        return {"bytes": w["bytes"] + 12 * case["n"] ** 3 + 12 * cells, "flops": w["flops"]}
    if kind == "refine3":
        # the coarse volume and about three refined samples per coarse cell
        coarse = case["cx"] * case["cy"] * case["cz"]
        w = _trace_work(4.0 * coarse, case["n"], case["n"] ** 3, 19)
        return {"bytes": w["bytes"] + 8.0 * coarse * 8 ** (case["levels"] - 1), "flops": w["flops"]}
    macs = 9.0 * (2 * 32 + 32 * 32 + 32)  # multiply-adds of the three layers per pixel
    if kind == "infer":
        p = case["nz"] * case["ny"] * case["nx"]
        return {"bytes": 20.0 * p, "flops": 2 * macs * p}
    p = case["batch"] * case["h"] * case["w"]
    # forward, weight gradients of all layers, data gradients of the upper two
    return {"bytes": 12.0 * p + 24.0 * qsl.QSL_CNN_NPARAMS, "flops": 2 * p * (2 * macs + 9 * (32 * 32 + 32))}


# ---------------------------------------------------------------- 64-bit values
def _exact_hyper(case, seed):
    """Closed forms of B = (lam x, -lam y, b0): the flow is (x e^(lam t), y
    e^(-lam t), b0 t); a line leaves through the top at t = 1 / b0 or through
    x = +-1 before; footpoint Q from the Jacobian of the boundary map, length
    by Gauss-Legendre quadrature of |B| dt."""
    lam, b0 = _hyper_constants(seed)
    m = case["m"]
    c = -1 + (torch.arange(m, dtype=torch.float64) + 0.5) * 2 / m
    y, x = torch.meshgrid(c, c, indexing="ij")
    t_side = torch.log(1 / x.abs()) / lam
    top = t_side >= 1 / b0
    te = torch.where(top, torch.full_like(x, 1 / b0), t_side)
    k = math.exp(lam / b0)
    q = torch.where(top, torch.full_like(x, k * k + 1 / (k * k)),
                    lam * (x * x + y * y) / b0 + b0 / (lam * x * x))
    nodes, weights = np.polynomial.legendre.leggauss(48)
    L = torch.zeros_like(x)
    for u, wt in zip(nodes, weights):
        s = te * (0.5 * (u + 1))
        L += wt * torch.sqrt((lam * x) ** 2 * torch.exp(2 * lam * s) + (lam * y) ** 2 * torch.exp(-2 * lam * s) + b0 ** 2)
    return {"q": q.reshape(-1), "length": (L * te * 0.5).reshape(-1), "faces": None, "status": None}


def _exact_weights(seed):
    p = torch.as_tensor(_params(seed)).cuda()
    out, o = [], 0
    for shape in ((32, 2, 3, 3), (32,), (32, 32, 3, 3), (32,), (1, 32, 3, 3), (1,)):
        n = math.prod(shape)
        v = p[o:o + n].view(shape)
        out.append((v.bfloat16() if len(shape) == 4 else v).double())  # the passes' weights are BF16
        o += n
    return out


def _exact_logits(X, w):
    conv = torch.nn.functional.conv2d
    a1 = torch.relu(conv(X, w[0], w[1], padding=1))
    a2 = torch.relu(conv(a1, w[2], w[3], padding=1))
    return conv(a2, w[4], w[5], padding=1)[:, 0]


def exact(case, seed):
    """None for the traced maps of charge fields: a 64-bit trace of every line
    through the gridded field in plain torch takes minutes."""
    kind = case["kind"]
    if kind == "hyper":
        return _exact_hyper(case, seed)
    if kind == "infer":
        X = _features64(*_coarse_volume(case, seed))
        w = _exact_weights(seed)
        prob = torch.cat([torch.sigmoid(_exact_logits(X[i:i + 4], w)) for i in range(0, X.shape[0], 4)])
        return {"X": X, "prob": prob}
    if kind == "train":
        X, Y, pos = _batch(case, seed)
        w = [v.requires_grad_(True) for v in _exact_weights(seed)]
        y = Y.double()
        z = _exact_logits(X.double(), w)
        sp = torch.nn.functional.softplus
        loss = (pos * y * sp(-z) + (1 - y) * sp(z)).mean()
        loss.backward()
        return {"loss": loss.detach().view(1), "grad": torch.cat([v.grad.reshape(-1) for v in w])}
    return None
