"""Performance cases: the work a lattice program has this library do, through
its public entry points, from the smallest calls to the largest lattices.

A case is a dict of plain values; ``kind`` names the call sequence:

* ``eo_op``       an even-odd operator applied ``times`` times to packed fields and
                  the result unpacked: a polynomial filter, a power iteration, a
                  step of an eigensolver.
* ``solve``       Mhat^+ Mhat x = b by CG (FP64 or mixed, one or many right-hand sides).
* ``batch``       the CG of many small lattices in one call (a volume or coupling scan).
* ``propagator``  D x = b with clover fermions for a new gauge field: clover field,
                  solve, canonical solution.
* ``gauge_md``    one leapfrog step of pure-gauge molecular dynamics.
* ``hmc``         one molecular-dynamics trajectory with two flavours.
* ``force``       the pseudofermion force, Wilson or clover, for a given solution.
* ``diff_dirac``  forward and backward of the differentiable D(U) psi.

Links have plaquette about 0.6 and no gauge fixing (random gauge-rotated
near-identity links), sources are Gaussian.  Such links are rougher than an
equilibrium field, so the bare masses here, 0.15 to 0.5, are the ones at which
a solve takes the 40 to 55 iterations it takes on an equilibrium field at -0.2.
"""

import math

import torch

from paper_2411_18511_gb300 import autograd, fields, hr
from paper_2411_18511_gb300.hmc import HMC

REP = {"fund": hr.HR_FUND, "adj": hr.HR_ADJ, "adjmat": hr.HR_ADJ_MAT}
PREC = {"f64": hr.HR_F64, "f32": hr.HR_F32, "f16": hr.HR_F16}
OP = {"hop": hr.HR_OP_HOP, "schur": hr.HR_OP_SCHUR, "schur_dag": hr.HR_OP_SCHUR_DAG, "normal": hr.HR_OP_NORMAL}
BATCH_EXTENTS = (8, 8, 10, 12, 12, 14, 16, 16, 18, 20, 22, 24)


def listed():
    return [
        # the benchmark workload: D_eo and D_oe of the whole 48^4 lattice, four times over, in the tuned shape
        {"name": "hop_fund_f64_48", "kind": "eo_op", "op": "hop", "rep": "fund", "prec": "f64", "times": 4,
         "t": 48, "l1": 48, "l2": 48, "l3": 48, "bc": 0, "n_rhs": 1, "tuned": True},
        # adjoint fermions (technicolour studies), antiperiodic time, as a program that never tunes calls it
        {"name": "normal_adj_f64_24", "kind": "eo_op", "op": "normal", "rep": "adj", "prec": "f64", "times": 2,
         "t": 32, "l1": 24, "l2": 24, "l3": 24, "bc": 1, "n_rhs": 1, "tuned": False},
        # the smallest production lattice: launches and latency are what counts
        {"name": "normal_fund_f64_8", "kind": "eo_op", "op": "normal", "rep": "fund", "prec": "f64", "times": 1,
         "t": 8, "l1": 8, "l2": 8, "l3": 8, "bc": 1, "n_rhs": 1, "tuned": False},
        # time to solution of the benchmark's CG size with the fastest inner precision
        {"name": "cg_f16_32", "kind": "solve", "rep": "fund", "inner": "f16", "delta": 3e-3, "n_rhs": 1, "m0": 0.2,
         "t": 32, "l1": 32, "l2": 32, "l3": 32, "bc": 0, "tuned": True},
        # propagators with many sources on a ragged lattice, FP32 inner
        {"name": "cg_f32_rhs16", "kind": "solve", "rep": "fund", "inner": "f32", "delta": 1e-5, "n_rhs": 16,
         "m0": 0.2, "t": 26, "l1": 22, "l2": 18, "l3": 20, "bc": 1, "tuned": False},
        # the twelve lattices of a finite-volume study in one call
        {"name": "batch_12", "kind": "batch", "n_lat": 12, "shift": 0, "m0": 0.2},
        # clover propagator: new gauge field, clover field, full solve
        {"name": "clover_solve_24", "kind": "propagator", "clover": "sw", "inner": "f32", "delta": 1e-5, "m0": 0.2,
         "c_sw": 1.0, "t": 24, "l1": 24, "l2": 24, "l3": 24, "bc": 1},
        # one step of pure-gauge molecular dynamics (thermalisation, quenched ensembles)
        {"name": "gauge_md_32", "kind": "gauge_md", "beta": 2.2, "eps": 0.05, "t": 32, "l1": 32, "l2": 32, "l3": 32},
        # a whole trajectory on two time scales, the schedule of the benchmark
        {"name": "hmc_16", "kind": "hmc", "inner": "f16", "delta": 0.01, "beta": 2.2, "m0": 0.2, "n_steps": 6,
         "n_gauge": 3, "tau": 1.0, "c_sw": 0.0, "hasenbusch": False, "t": 16, "l1": 16, "l2": 16, "l3": 16},
        # the molecular-dynamics force of two Wilson flavours
        {"name": "force_32", "kind": "force", "clover": "none", "m0": 0.2, "c_sw": 0.0, "t": 32, "l1": 32, "l2": 32,
         "l3": 32, "bc": 1},
        # the clover force with its determinant, on an odd-shaped lattice
        {"name": "clover_force_20", "kind": "force", "clover": "sw", "m0": 0.2, "c_sw": 1.0, "t": 20, "l1": 14,
         "l2": 18, "l3": 22, "bc": 1},
        # a differentiable Dirac application in a training loop: packing, D, gradients of links and spinor
        {"name": "diff_dirac_16", "kind": "diff_dirac", "m0": 0.2, "t": 16, "l1": 16, "l2": 16, "l3": 16, "bc": 1},
    ]


# ---------------------------------------------------------------- drawn cases

def _extents(rng, vmin, vmax, lo=4, hi=48):
    """Even extents with a volume spread over the logarithm of [vmin, vmax], rarely hypercubic."""
    target = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    for _ in range(200):
        side = target ** 0.25
        d = [max(lo, min(hi, 2 * round(side * math.exp(rng.uniform(-0.4, 0.4)) / 2))) for _ in range(4)]
        v = d[0] * d[1] * d[2] * d[3]
        if 0.6 * target <= v <= 1.6 * target and v <= vmax:
            return dict(zip(("t", "l1", "l2", "l3"), d))
    n = 2 * max(2, int(side // 2))
    return {"t": n, "l1": n, "l2": n, "l3": n}


def draw(rng):
    kind = rng.choice(["eo_op", "eo_op", "eo_op", "solve", "solve", "batch", "propagator", "gauge_md", "hmc", "force",
                       "force", "diff_dirac"])
    m0 = round(rng.uniform(0.15, 0.5), 3)
    bc = rng.choice([0, 1, 1, 15])
    if kind == "eo_op":
        rep = rng.choice(["fund", "fund", "fund", "adj", "adjmat"])
        n_rhs = rng.choice([1, 1, 1, 2, 8])
        vmax = 48 ** 4 // ((2 if rep == "fund" else 6) * n_rhs)
        return {"kind": kind, "op": rng.choice(list(OP)), "rep": rep, "prec": rng.choice(["f64", "f64", "f32", "f16"]),
                "times": rng.choice([1, 2]), **_extents(rng, 4 ** 4, vmax), "bc": bc, "n_rhs": n_rhs, "tuned": False}
    if kind == "solve":
        inner = rng.choice(["f64", "f32", "f16"])
        n_rhs = rng.choice([1, 1, 4, 16])
        rep = rng.choice(["fund", "fund", "adj"])
        return {"kind": kind, "rep": rep, "inner": inner, "delta": {"f64": 0.1, "f32": 1e-5, "f16": 1e-2}[inner],
                "n_rhs": n_rhs, "m0": m0, **_extents(rng, 6 ** 4, 28 ** 4 // n_rhs), "bc": bc, "tuned": False}
    if kind == "batch":
        return {"kind": kind, "n_lat": rng.randint(2, 10), "shift": rng.randint(0, 11), "m0": m0}
    if kind == "propagator":
        inner = rng.choice(["f64", "f32", "f16"])
        return {"kind": kind, "clover": rng.choice(["sw", "exp"]), "inner": inner,
                "delta": {"f64": 0.1, "f32": 1e-5, "f16": 1e-2}[inner], "m0": m0,
                "c_sw": round(rng.uniform(0.5, 1.3), 2), **_extents(rng, 6 ** 4, 20 ** 4), "bc": bc}
    if kind == "gauge_md":
        return {"kind": kind, "beta": round(rng.uniform(2.0, 2.6), 2), "eps": round(rng.uniform(0.02, 0.2), 3),
                **_extents(rng, 4 ** 4, 40 ** 4)}
    if kind == "hmc":
        n = rng.choice([1, 3])
        c_sw, heavy = rng.choice([0.0, 0.0, 1.0]), rng.choice([False, True])
        dear = heavy or c_sw > 0.0
        return {"kind": kind, "inner": rng.choice(["f64", "f32", "f16"]), "delta": 0.01, "beta": 2.2, "m0": m0,
                "n_steps": 2 if dear else rng.choice([2, 4]), "n_gauge": n, "tau": 0.5, "c_sw": c_sw,
                "hasenbusch": heavy, **_extents(rng, 6 ** 4, (12 if dear else 16) ** 4, hi=24)}
    if kind == "force":
        clover = rng.choice(["none", "sw", "exp"])
        vmax = {"none": 40, "sw": 24, "exp": 18}[clover] ** 4
        return {"kind": kind, "clover": clover, "m0": m0, "c_sw": 0.0 if clover == "none" else 1.0,
                **_extents(rng, 4 ** 4, vmax), "bc": bc}
    return {"kind": kind, "m0": m0, **_extents(rng, 4 ** 4, 32 ** 4), "bc": bc}


# ---------------------------------------------------------------- inputs

def _dims(case):
    return case["t"], case["l1"], case["l2"], case["l3"]


def _vol(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _qmul(a, b):
    """(a0 + i a.s)(b0 + i b.s), quaternions in the last axis."""
    a0, a1, a2, a3 = a.unbind(-1)
    b0, b1, b2, b3 = b.unbind(-1)
    return torch.stack((a0 * b0 - a1 * b1 - a2 * b2 - a3 * b3,
                        a0 * b1 + b0 * a1 - (a2 * b3 - a3 * b2),
                        a0 * b2 + b0 * a2 - (a3 * b1 - a1 * b3),
                        a0 * b3 + b0 * a3 - (a1 * b2 - a2 * b1)), -1)


def _qconj(a):
    return a * torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=a.dtype, device=a.device)


def _links(dims, gen):
    """Canonical links [4, V, 4]: near-identity SU(2) elements (plaquette about
    0.6) in a random gauge, so that single links are spread over the group."""
    def unit(q):
        return q / q.norm(dim=-1, keepdim=True)

    def normal(*shape):
        return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)

    q = 0.31 * normal(4, *dims, 4)
    q[..., 0] = 1.0
    q = unit(q)
    rot = unit(normal(*dims, 4))
    for mu in range(4):
        q[mu] = _qmul(_qmul(rot, q[mu]), _qconj(torch.roll(rot, -1, mu)))
    return unit(q).reshape(4, _vol(dims), 4).contiguous()


def _spinor(dims, nc, gen, n_rhs=1):
    shape = ((n_rhs,) if n_rhs > 1 else ()) + (_vol(dims), 4, nc)
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=gen) * math.sqrt(2.0)


def _even(dims):
    c = [torch.arange(n, device="cuda") for n in dims]
    s = c[0][:, None, None, None] + c[1][:, None, None] + c[2][:, None] + c[3]
    return (s % 2 == 0).reshape(-1)


def _opts(case, n_rhs=1):
    o = hr.hr_solver_default_opts()
    o.inner_prec = PREC[case["inner"]]
    o.reliable_delta = case["delta"]
    o.n_rhs = n_rhs
    return o


_tuned = set()


def _tune(ctx, dims, rep, prec, n_rhs, q, psi):
    """A program tunes a configuration once, when it starts."""
    key = (tuple(dims), rep, prec, n_rhs)
    if key in _tuned:
        return
    _tuned.add(key)
    gauge = fields.pack_gauge(ctx, dims, rep, prec, q)
    src = fields.pack_spinor(ctx, dims, rep, prec, hr.HR_ODD, psi)
    dst = fields.empty_spinor(dims, rep, prec, hr.HR_EVEN, n_rhs)
    hr.hr_autotune_hop(ctx, dims, rep, prec, hr.HR_EVEN, n_rhs, gauge, src, dst, reps=10)


def _batch_dims(case):
    n = len(BATCH_EXTENTS)
    return [(e, e, e, e) for e in (BATCH_EXTENTS[(case["shift"] + k) % n] for k in range(case["n_lat"]))]


def _inputs(case, seed):
    """The seeded canonical inputs shared by prepare() and exact()."""
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        out = []
        for d in _batch_dims(case):
            q = _links(d, gen)
            out.append((q, _spinor(d, 2, gen)))
        return out
    dims = _dims(case)
    q = _links(dims, gen)
    if kind == "eo_op":
        return q, _spinor(dims, 2 if case["rep"] == "fund" else 3, gen, case["n_rhs"])
    if kind == "solve":
        return q, _spinor(dims, 2 if case["rep"] == "fund" else 3, gen, case["n_rhs"])
    if kind in ("propagator", "diff_dirac"):
        return q, _spinor(dims, 2, gen), _spinor(dims, 2, gen)
    mom = torch.randn((4, _vol(dims), 3), dtype=torch.float64, device="cuda", generator=gen)
    if kind == "gauge_md":
        return q, mom
    return q, mom, _spinor(dims, 2, gen), _spinor(dims, 2, gen)


def prepare(case, seed):
    ctx = autograd.default_context()
    kind = case["kind"]
    if kind == "batch":
        dims = _batch_dims(case)
        gauges, bs, xs = [], [], []
        for d, (q, b) in zip(dims, _inputs(case, seed)):
            gauges.append(fields.pack_gauge(ctx, d, hr.HR_FUND, hr.HR_F64, q))
            bs.append(fields.pack_spinor(ctx, d, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, b))
            xs.append(fields.zeros_spinor(d, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN))
        opts = hr.hr_solver_default_opts()
        work = fields.empty_bytes(hr.hr_cg_batch_workspace_bytes(dims, hr.HR_FUND))
        return dict(case=case, ctx=ctx, dims=dims, gauges=gauges, bs=bs, xs=xs, opts=opts, work=work)
    dims = hr.Lattice(_dims(case), case.get("bc", 0))
    st = dict(case=case, ctx=ctx, dims=dims)
    if kind == "eo_op":
        q, psi = _inputs(case, seed)
        rep, prec, n = REP[case["rep"]], PREC[case["prec"]], case["n_rhs"]
        if case["tuned"]:
            _tune(ctx, dims, rep, prec, n, q, psi)
        st["gauge"] = fields.pack_gauge(ctx, dims, rep, prec, q)
        if case["op"] == "hop":
            st["src"] = fields.pack_spinor(ctx, dims, rep, prec, hr.HR_FULL, psi)
            st["tmp"] = [fields.empty_spinor(dims, rep, prec, hr.HR_FULL, n) for _ in range(2)]
        else:
            st["src"] = fields.pack_spinor(ctx, dims, rep, prec, hr.HR_EVEN, psi)
            st["tmp"] = [fields.empty_spinor(dims, rep, prec, hr.HR_EVEN, n) for _ in range(2)]
        st["work"] = fields.empty_bytes(hr.hr_dirac_workspace_bytes(dims, rep, prec, OP[case["op"]], n))
    elif kind == "solve":
        q, b = _inputs(case, seed)
        rep, n = REP[case["rep"]], case["n_rhs"]
        if case["tuned"]:
            for prec in (hr.HR_F64, hr.HR_F32, hr.HR_F16):
                _tune(ctx, dims, rep, prec, n, q, b)
        st["gauge"] = fields.pack_gauge(ctx, dims, rep, hr.HR_F64, q)
        st["b"] = fields.pack_spinor(ctx, dims, rep, hr.HR_F64, hr.HR_EVEN, b)
        st["x"] = fields.zeros_spinor(dims, rep, hr.HR_F64, hr.HR_EVEN, n)
        st["opts"] = _opts(case, n)
        st["work"] = fields.empty_bytes(hr.hr_cg_workspace_bytes(dims, rep, st["opts"]))
    elif kind == "propagator":
        q, b, _ = _inputs(case, seed)
        st["q"] = q
        st["b"] = fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, b)
        st["x"] = fields.zeros_spinor(dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL)
        st["opts"] = _opts(case)
        st["work"] = fields.empty_bytes(
            hr.hr_solve_full_clover_workspace_bytes(dims, hr.HR_FUND, st["opts"], hr.HR_SYSTEM_D))
        st["clover"] = fields.empty_bytes(hr.hr_clover_packed_bytes(dims, hr.HR_FUND, hr.HR_F64))
    elif kind == "gauge_md":
        st["q"], st["mom"] = _inputs(case, seed)
    elif kind == "hmc":
        dims = st["dims"] = hr.Lattice(_dims(case), 1)
        q = _inputs(case, seed)[0]
        chain = HMC(ctx, dims, case["beta"], case["m0"], True, case["n_steps"], case["tau"], solver=_opts(case),
                    seed=seed, m0_hasenbusch=case["m0"] + 0.4 if case["hasenbusch"] else None,
                    n_steps_gauge=case["n_gauge"], c_sw=case["c_sw"] or None)
        pf = chain.draw_pseudofermion(q)
        eta, phi = pf if case["hasenbusch"] else (pf, None)
        st.update(q=q, mom=chain.draw_momenta(), prm=chain.prm, eta=eta, phi=phi, work=chain.work)
    elif kind == "force":
        q, _, x, _ = _inputs(case, seed)
        st["q"] = q
        st["gauge"] = fields.pack_gauge(ctx, dims, hr.HR_FUND, hr.HR_F64, q)
        st["x"] = fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, x)
        if case["clover"] == "none":
            st["work"] = fields.empty_bytes(hr.hr_fermion_force_workspace_bytes(dims))
        else:
            st["kind"] = hr.HR_CLOVER_SW if case["clover"] == "sw" else hr.HR_CLOVER_EXP
            st["clover"] = fields.build_clover(ctx, dims, hr.HR_FUND, hr.HR_F64, st["kind"], case["m0"],
                                               case["c_sw"], q)
            st["work"] = fields.empty_bytes(hr.hr_clover_force_workspace_bytes(dims))
    elif kind == "diff_dirac":
        st["q"], st["psi"], st["g"] = _inputs(case, seed)
    return st


# ---------------------------------------------------------------- one pass

def run(st):
    return globals()["_run_" + st["case"]["kind"]](st)


def _run_eo_op(st):
    case, ctx, dims = st["case"], st["ctx"], st["dims"]
    rep, prec, n, op = REP[case["rep"]], PREC[case["prec"]], case["n_rhs"], OP[case["op"]]
    src = st["src"]
    for k in range(case["times"]):
        dst = st["tmp"][k % 2]
        if op == hr.HR_OP_HOP:
            half = src.numel() // 2
            hr.hr_dirac_eo(ctx, dims, 0.0, rep, prec, hr.HR_EVEN, op, n, st["gauge"], src[half:], dst[:half])
            hr.hr_dirac_eo(ctx, dims, 0.0, rep, prec, hr.HR_ODD, op, n, st["gauge"], src[:half], dst[half:])
        else:
            hr.hr_dirac_eo(ctx, dims, -0.2, rep, prec, hr.HR_EVEN, op, n, st["gauge"], src, dst, st["work"])
        src = dst
    out = fields.unpack_spinor(ctx, dims, rep, prec, hr.HR_FULL if op == hr.HR_OP_HOP else hr.HR_EVEN, src, n)
    # a program that computes in FP32 or binary16 goes on in that type
    if case["prec"] == "f32":
        return out.to(torch.complex64)
    return torch.view_as_real(out).to(torch.float16) if case["prec"] == "f16" else out


def _run_solve(st):
    case, dims, rep = st["case"], st["dims"], REP[st["case"]["rep"]]
    hr.hr_cg_solve(st["ctx"], dims, case["m0"], rep, st["opts"], st["gauge"], st["b"], st["x"], st["work"])
    return fields.unpack_spinor(st["ctx"], dims, rep, hr.HR_F64, hr.HR_EVEN, st["x"], case["n_rhs"])


def _run_batch(st):
    hr.hr_cg_solve_batch(st["ctx"], st["dims"], st["case"]["m0"], hr.HR_FUND, st["opts"], st["gauges"], st["bs"],
                         st["xs"], st["work"])
    return [fields.unpack_spinor(st["ctx"], d, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, x)
            for d, x in zip(st["dims"], st["xs"])]


def _run_propagator(st):
    case, ctx, dims = st["case"], st["ctx"], st["dims"]
    kind = hr.HR_CLOVER_SW if case["clover"] == "sw" else hr.HR_CLOVER_EXP
    gauge = fields.pack_gauge(ctx, dims, hr.HR_FUND, hr.HR_F64, st["q"])
    hr.hr_clover_build(ctx, dims, hr.HR_FUND, hr.HR_F64, kind, case["m0"], case["c_sw"], st["q"], st["clover"])
    hr.hr_solve_full_clover(ctx, dims, hr.HR_FUND, st["opts"], hr.HR_SYSTEM_D, gauge, st["clover"], st["b"], st["x"],
                            st["work"])
    return fields.unpack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, st["x"])


def _run_gauge_md(st):
    case, ctx, dims = st["case"], st["ctx"], st["dims"]
    q, mom = st["q"].clone(), st["mom"].clone()
    force = torch.zeros_like(mom)
    hr.hr_gauge_force(ctx, dims, case["beta"], q, 1.0, force)
    hr.hr_mom_update(ctx, dims, 0.5 * case["eps"], force, mom)
    hr.hr_link_update(ctx, dims, case["eps"], mom, q)
    force.zero_()
    hr.hr_gauge_force(ctx, dims, case["beta"], q, 1.0, force)
    hr.hr_mom_update(ctx, dims, 0.5 * case["eps"], force, mom)
    return q, mom


def _run_hmc(st):
    q, mom = st["q"].clone(), st["mom"].clone()
    hr.hr_hmc_trajectory(st["ctx"], st["dims"], st["prm"], q, mom, st["eta"], st["work"], phi=st["phi"])
    return q, mom


def _run_force(st):
    case, ctx, dims = st["case"], st["ctx"], st["dims"]
    force = torch.zeros((4, _vol(dims), 3), dtype=torch.float64, device="cuda")
    if case["clover"] == "none":
        hr.hr_fermion_force(ctx, dims, case["m0"], hr.HR_FUND, st["gauge"], st["x"], None, -1.0, force, st["work"])
    else:
        hr.hr_clover_fermion_force(ctx, dims, case["m0"], case["c_sw"], st["q"], st["gauge"], st["clover"], st["x"],
                                   True, 1.0, force, st["work"], kind=st["kind"])
    return force


def _run_diff_dirac(st):
    q, psi = st["q"].detach().requires_grad_(True), st["psi"].detach().requires_grad_(True)
    y = autograd.DiracApply.apply(q, psi, st["dims"], st["case"]["m0"])
    gq, gpsi = torch.autograd.grad(y, (q, psi), st["g"])
    return y.detach(), gq, gpsi


# ---------------------------------------------------------------- the work that a pass cannot do without

def _hop_bytes(rep, prec):
    """Spinor in and out, eight links: bytes per output site of one hop."""
    nc = 2 if rep == "fund" else 3
    real = {"f64": 8, "f32": 4, "f16": 2}[prec]
    scale = 4 if prec == "f16" else 0
    return 2 * (8 * nc * real + scale), 8 * real * (9 if rep == "adjmat" else 4)


def _op_work(vh, rep, prec, op, n=1):
    """One application of an even-odd operator on vh sites and n right-hand sides (hop: both parities)."""
    sp, links = _hop_bytes(rep, prec)
    hops = {"hop": 2, "schur": 2, "schur_dag": 2, "normal": 4}[op]
    flops = hops * n * vh * (624 if rep == "fund" else 744)
    aux = 0 if op == "hop" else hops // 2 * sp // 2
    return vh * (hops * (links + n * sp) + n * aux), flops


CG_ITERS = 47  # iterations to 1e-10 at m0 = 0.2 and this plaquette


def _cg_work(vh, rep, inner, n, iters=CG_ITERS):
    b, f = _op_work(vh, rep, inner, "normal", n)
    half = _hop_bytes(rep, inner)[0] // 2
    return iters * (b + 7 * n * vh * half), iters * (f + 6 * n * vh * (32 if rep == "fund" else 48))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_cg_work(_vol(d) // 2, "fund", "f64", 1) for d in _batch_dims(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    V = _vol(_dims(case))
    vh, spin, gauge, mom = V // 2, V * 128, 4 * V * 32, 4 * V * 24
    if kind == "eo_op":
        b, f = _op_work(vh, case["rep"], case["prec"], case["op"], case["n_rhs"])
        full = 1 if case["op"] == "hop" else 0.5
        sp = _hop_bytes(case["rep"], case["prec"])[0] // 2
        out = case["n_rhs"] * V * (full * sp + (128 if case["rep"] == "fund" else 192))
        return {"bytes": case["times"] * b + out, "flops": case["times"] * f}
    if kind == "solve":
        b, f = _cg_work(vh, case["rep"], case["inner"], case["n_rhs"])
        return {"bytes": b, "flops": f}
    if kind == "propagator":
        b, f = _cg_work(vh, "fund", case["inner"], 1)
        clover = 2 * gauge + V * 512  # links in, packed links and clover field out
        return {"bytes": b + clover + 2 * spin, "flops": f + V * 6 * 12 * 28}
    if kind == "gauge_md":  # two forces, one link update, two momentum updates
        return {"bytes": 2 * (gauge + mom) + 2 * gauge + mom + 2 * 3 * mom, "flops": 4 * V * (2 * 13 * 28 + 60)}
    if kind == "hmc":
        solves = (2 * case["n_steps"] + 1) * (2 if case["hasenbusch"] else 1) + 1
        b, f = _cg_work(vh, "fund", case["inner"], 1)
        md = 2 * case["n_steps"] * max(1, case["n_gauge"]) * 2
        return {"bytes": solves * (b + 4 * spin + gauge + mom) + md * (3 * gauge + 4 * mom),
                "flops": solves * (f + V * 4 * 300) + md * 4 * V * (13 * 28 + 60)}
    if kind == "force":
        b, f = _op_work(vh, "fund", "f64", "normal")
        extra = V * 256 if case["clover"] == "none" else V * (256 + 256 + 6 * 24) + 2 * gauge
        return {"bytes": b + extra + gauge + mom, "flops": f + V * 4 * (300 if case["clover"] == "none" else 1800)}
    # diff_dirac: D twice, the link gradient, every canonical tensor once
    b, f = _op_work(vh, "fund", "f64", "hop")
    return {"bytes": 2 * b + 2 * gauge + 4 * spin + spin, "flops": 2 * f + V * 4 * 250}


# ---------------------------------------------------------------- the same results in 64 bits, from the definitions

def _umat(q, rep):
    """Link matrices [..., nc, nc] of quaternions [..., 4]."""
    a0, a1, a2, a3 = q.unbind(-1)
    if rep == "fund":
        return torch.stack((torch.complex(a0, a3), torch.complex(a2, a1), torch.complex(-a2, a1),
                            torch.complex(a0, -a3)), -1).unflatten(-1, (2, 2))
    w = a0 * a0 - a1 * a1 - a2 * a2 - a3 * a3
    rows = [w + 2 * a1 * a1, 2 * (a1 * a2 + a0 * a3), 2 * (a1 * a3 - a0 * a2),
            2 * (a1 * a2 - a0 * a3), w + 2 * a2 * a2, 2 * (a2 * a3 + a0 * a1),
            2 * (a1 * a3 + a0 * a2), 2 * (a2 * a3 - a0 * a1), w + 2 * a3 * a3]
    return torch.stack(rows, -1).unflatten(-1, (3, 3)).to(torch.complex128)


def _gammas():
    s = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128)
    z, e = torch.zeros((2, 2), dtype=torch.complex128), torch.eye(2, dtype=torch.complex128)
    g = [torch.cat((torch.cat((z, e), 1), torch.cat((e, z), 1)))]
    g += [torch.cat((torch.cat((z, -1j * k), 1), torch.cat((1j * k, z), 1))) for k in s]
    return g


class _Wilson:
    """The Wilson hopping term of canonical links q [4, V, 4], from its definition."""

    def __init__(self, q, dims, rep, bc):
        self.dims = tuple(dims)
        U = _umat(q, rep).reshape(4, *self.dims, *(2 * (2 if rep == "fund" else 3,)))
        sign = torch.ones((4, *self.dims, 1, 1), dtype=torch.float64, device=q.device)
        for mu in range(4):
            if (bc >> mu) & 1:
                sign[mu].select(mu, self.dims[mu] - 1).neg_()
        self.U = U * sign
        # rows of gamma_mu: gamma_mu psi = phase * psi[perm]
        self.g = []
        for m in _gammas():
            perm = m.abs().argmax(1)
            self.g.append((perm.tolist(), [complex(m[r, int(c)]) for r, c in enumerate(perm)]))

    @staticmethod
    def _mul(U, psi, dag):
        """U psi (or U^+ psi), psi [..., 4, nc]."""
        nc = U.shape[-1]
        cols = []
        for a in range(nc):
            acc = 0
            for b in range(nc):
                u = U[..., b, a].conj() if dag else U[..., a, b]
                acc = acc + u.unsqueeze(-1) * psi[..., b]
            cols.append(acc)
        return torch.stack(cols, -1)

    def _spin(self, mu, psi, sgn):
        perm, ph = self.g[mu]
        return torch.stack([psi[..., s, :] + sgn * ph[s] * psi[..., perm[s], :] for s in range(4)], -2)

    def hop(self, psi):
        """H psi of psi [V, 4, nc]."""
        p = psi.reshape(*self.dims, 4, -1)
        out = 0
        for mu in range(4):
            out = out + self._spin(mu, self._mul(self.U[mu], torch.roll(p, -1, mu), False), -1.0)
            out = out + self._spin(mu, torch.roll(self._mul(self.U[mu], p, True), 1, mu), 1.0)
        return out.reshape(psi.shape)


def _g5(psi):
    return psi * torch.tensor([-1.0, -1.0, 1.0, 1.0], dtype=torch.float64, device=psi.device)[:, None]


def _clover_matrix(q, dims, kind, m0, c_sw):
    """The site term A as two chiral 4 x 4 blocks [V, 2, 4, 4]."""
    Q = q.reshape(4, *dims, 4)
    g = [m.to(q.device) for m in _gammas()]
    C = 0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            a, b = Q[mu], torch.roll(Q[nu], -1, mu)
            c, d = _qconj(torch.roll(Q[mu], -1, nu)), _qconj(Q[nu])
            # the plaquette of each corner x, traversed from x, mu first
            p = _qmul(_qmul(a, b), _qmul(c, d))
            p1 = torch.roll(_qmul(_qmul(b, c), _qmul(d, a)), 1, mu)
            p2 = torch.roll(_qmul(_qmul(c, d), _qmul(a, b)), (1, 1), (mu, nu))
            p3 = torch.roll(_qmul(_qmul(d, a), _qmul(b, c)), 1, nu)
            v = (p + p1 + p2 + p3)[..., 1:] / 4.0  # F = (Q - Q^+) / 8 = (i / 4) vec(Q).s
            zero = torch.zeros_like(v[..., :1])
            F = _umat(torch.cat((zero, v), -1), "fund")
            s = 0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])
            blocks = torch.stack((s[:2, :2], s[2:, 2:]))
            C = C + 0.5j * torch.einsum("bst,...cd->...bsctd", blocks, F)
    C = C.reshape(-1, 2, 4, 4)
    A = 4.0 + m0
    if kind == "exp":
        return A * torch.linalg.matrix_exp(c_sw * C / A)
    return A * torch.eye(4, dtype=torch.complex128, device=q.device) + c_sw * C


def _site(A, psi):
    """A psi with A [V, 2, 4, 4], psi [V, 4, 2]."""
    return torch.einsum("vbij,vbj->vbi", A, psi.reshape(-1, 2, 4)).reshape(psi.shape)


def _cg(op, b, tol=1e-14, maxiter=400):
    """CG per leading index of b [n, V, 4, nc]; op acts on one field."""
    out = []
    for rhs in b:
        x, r = torch.zeros_like(rhs), rhs.clone()
        p, rr = r.clone(), float(r.abs().square().sum())
        bb = rr
        for _ in range(maxiter):
            if rr <= tol * tol * bb:
                break
            q = op(p)
            a = rr / float(torch.vdot(p.reshape(-1), q.reshape(-1)).real)
            x += a * p
            r -= a * q
            new = float(r.abs().square().sum())
            p = r + (new / rr) * p
            rr = new
        out.append(x)
    return torch.stack(out)


def _exact_solve(q, b, dims, rep, bc, m0):
    W, A = _Wilson(q, dims, rep, bc), 4.0 + m0
    mhat = lambda v: A * v - W.hop(W.hop(v)) / (4.0 * A)  # noqa: E731
    b = b * _even(dims)[:, None, None]
    return _cg(lambda v: _g5(mhat(_g5(mhat(v)))), b)


def _su2_derivative(q, dq):
    """d/dw_a under U -> exp(i w.s/2) U of a function with gradient dq in the quaternion components."""
    out = []
    for a in range(3):
        e = torch.zeros(4, dtype=q.dtype, device=q.device)
        e[a + 1] = 0.5
        out.append((_qmul(e.expand_as(q), q) * dq).sum(-1))
    return torch.stack(out, -1)


def _gauge_force(q, dims, beta):
    Q = q.reshape(4, *dims, 4)
    F = []
    for mu in range(4):
        S = 0
        for nu in range(4):
            if nu == mu:
                continue
            up = _qmul(_qmul(torch.roll(Q[nu], -1, mu), _qconj(torch.roll(Q[mu], -1, nu))), _qconj(Q[nu]))
            dn = _qmul(_qmul(_qconj(torch.roll(Q[nu], -1, mu)), _qconj(Q[mu])), Q[nu])
            S = S + up + torch.roll(dn, 1, nu)
        F.append(0.5 * beta * _qmul(Q[mu], S)[..., 1:])
    return torch.stack(F).reshape(4, -1, 3)


def exact(case, seed):
    kind = case["kind"]
    if kind == "hmc":
        return None  # some hundred thousand hops
    if kind == "batch":
        return [_exact_solve(q, b[None], d, "fund", 0, case["m0"])[0]
                for d, (q, b) in zip(_batch_dims(case), _inputs(case, seed))]
    dims, bc = _dims(case), case.get("bc", 0)
    if kind == "eo_op":
        if case["n_rhs"] * case["times"] * _vol(dims) > 6 * 48 ** 4:
            return None
        q, psi = _inputs(case, seed)
        W, out = _Wilson(q, dims, case["rep"], bc), []
        for v in psi if case["n_rhs"] > 1 else psi[None]:
            A = 4.0 - 0.2
            mhat = lambda u: A * u - W.hop(W.hop(u)) / (4.0 * A)  # noqa: E731
            if case["op"] != "hop":
                v = v * _even(dims)[:, None, None]
            for _ in range(case["times"]):
                if case["op"] == "hop":
                    v = -0.5 * W.hop(v)
                elif case["op"] == "schur":
                    v = mhat(v)
                elif case["op"] == "schur_dag":
                    v = _g5(mhat(_g5(v)))
                else:
                    v = _g5(mhat(_g5(mhat(v))))
            out.append(v)
        return torch.stack(out) if case["n_rhs"] > 1 else out[0]
    if kind == "solve":
        if case["n_rhs"] * _vol(dims) > 1.5 * 32 ** 4:
            return None
        q, b = _inputs(case, seed)
        x = _exact_solve(q, b if case["n_rhs"] > 1 else b[None], dims, case["rep"], bc, case["m0"])
        return x if case["n_rhs"] > 1 else x[0]
    if kind == "propagator":
        q, b, _ = _inputs(case, seed)
        W = _Wilson(q, dims, "fund", bc)
        A = _clover_matrix(q, dims, case["clover"], case["m0"], case["c_sw"])
        D = lambda v: _site(A, v) - 0.5 * W.hop(v)  # noqa: E731
        ddag = lambda v: _g5(D(_g5(v)))  # noqa: E731
        return _cg(lambda v: ddag(D(v)), ddag(b)[None], maxiter=600)[0]
    if kind == "gauge_md":
        q, mom = _inputs(case, seed)
        mom = mom - 0.5 * case["eps"] * _gauge_force(q, dims, case["beta"])
        nrm = mom.norm(dim=-1, keepdim=True)
        th = 0.5 * case["eps"] * nrm
        q = _qmul(torch.cat((torch.cos(th), torch.sin(th) * mom / nrm), -1), q)
        q = q / q.norm(dim=-1, keepdim=True)
        return q, mom - 0.5 * case["eps"] * _gauge_force(q, dims, case["beta"])
    if kind == "force":
        q, _, x, _ = _inputs(case, seed)
        even = _even(dims)[:, None, None]
        x, A = x * even, 4.0 + case["m0"]
        q = q.requires_grad_(True)
        W = _Wilson(q, dims, "fund", bc)
        if case["clover"] == "none":
            y = A * x - W.hop(W.hop(x)) / (4.0 * A)
            f = -y.abs().square().sum()
        else:
            M = _clover_matrix(q, dims, case["clover"], case["m0"], case["c_sw"])
            t = torch.linalg.solve(M, W.hop(x).reshape(-1, 2, 4, 1)).reshape(x.shape)
            y = _site(M, x) - 0.25 * W.hop(t)
            f = -2.0 * (y.detach().conj() * y).real.sum()
            if case["clover"] == "sw":
                f = f - 2.0 * torch.linalg.slogdet(M[~_even(dims)])[1].sum()
        (dq,) = torch.autograd.grad(f, q)
        return _su2_derivative(q.detach(), dq)
    q, psi, g = _inputs(case, seed)
    q, psi = q.requires_grad_(True), psi.requires_grad_(True)
    y = (4.0 + case["m0"]) * psi - 0.5 * _Wilson(q, dims, "fund", bc).hop(psi)
    gq, gpsi = torch.autograd.grad(y, (q, psi), g)
    return y.detach(), gq, gpsi
