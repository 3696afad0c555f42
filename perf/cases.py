"""The measured cases: what a user of the library has it do, through its Python entry points.

Each case is a dict of plain values with a "kind":

* ``field``   density and Poisson solve of a held state: the diagnostic a caller
  polls between steps (a few dozen small launches);
* ``gemm``    one dense contraction in one of the precision modes;
* ``create``  dense f on the grid -> MPS -> dense f (encode and decode);
* ``stage``   one explicit Euler stage that a caller composes from the operator,
  the addition and the compression;
* ``run``     host grid in, host grid and records out (``Context.run``);
* ``step``    one RK4 step of a resident simulation, its new f and its records;
* ``multi``   the same for electrons and ions on one field, with collisions;
* ``group``   one step of many resident simulations of mixed sizes.

States are compared as dense f on the grid: the cores themselves are unique only
up to an orthogonal change of basis on every bond.  ``exact`` does the same
arithmetic on the full grid in numpy (finite differences, RK4, and successive
SVDs of the unfoldings for every truncation to a bond cap); the intermediate
compressions of a step, to a relative 1e-10 per bond, are the identity there.
The truncation error of the records is left out: where no bond reaches the cap it
is the rounding of what was cut at 1e-10.
"""
import math

import numpy as np
import torch

from paper_2205_11990_gb300 import inputs, vpmps

SEQ, IF, S2, S3 = inputs.SEQ, inputs.INTERLEAVED, inputs.SEQ_S2, inputs.SEQ_S3
TOL = 1e-10
MODES = 32  # separable perturbation modes of a saturated state (rank 65 at the x / v cut)

_ctx = None


def _context():
    """The one context of a user's program (its workspaces are kept between calls)."""
    global _ctx
    if _ctx is None:
        _ctx = vpmps.Context()
    return _ctx


# --------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: charge density and field of a 64 x 64 state, polled between steps
        dict(name="field_64", kind="field", nx=6, nv=6, mapping=SEQ, chi=16),
        # a contraction of the sweeps' size (R times the next core), ragged in every dimension
        dict(name="gemm_fp64", kind="gemm", M=341, N=1008, K=503, precision="fp64"),
        # the tensor-core mode that keeps FP32 accuracy
        dict(name="gemm_tf32x3", kind="gemm", M=512, N=1008, K=504, precision="tf32x3"),
        # a dense 1024 x 1024 f encoded at the bond cap of the two-stream workload and decoded again
        dict(name="create_1024", kind="create", nx=10, nv=10, mapping=SEQ, chi=64),
        # a caller's own stage (operator, addition, compression) on a ragged interleaved grid
        dict(name="stage_if_128x64", kind="stage", nx=7, nv=6, mapping=IF, chi=24),
        # the whole call of a small run, host to host, on the default path: Landau-sized grid
        dict(name="run_64", kind="run", nx=6, nv=6, mapping=SEQ, chi=16, steps=2, modes=6),
        # one step at the ordinary sizes: 256 x 256 (one sim, default streams) ...
        dict(name="step_256", kind="step", nx=8, nv=8, mapping=SEQ, chi=32, streams=2),
        # ... the interleaved ordering, whose field term makes large bonds ...
        dict(name="step_if_128", kind="step", nx=7, nv=7, mapping=IF, chi=32, streams=0),
        # ... the benchmark workload, saturated two-stream 1024 x 1024 at chi = 64 ...
        dict(name="step_1024", kind="step", nx=10, nv=10, mapping=SEQ, chi=64, streams=0),
        # ... and the largest configuration, 4096 x 4096 at chi = 128
        dict(name="step_4096", kind="step", nx=12, nv=12, mapping=SEQ, chi=128, streams=0, modes=64),
        # electrons and ions on the Buneman grids (S3), with collisions
        dict(name="multi_512", kind="multi", nx=9, nv=9, mapping=S3, chi=64),
        # many small runs stepped together (batching, serving)
        dict(name="group_16", kind="group", members=16, low=6, high=8, chi=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["field", "gemm", "gemm", "create", "stage", "run", "step", "step", "step", "multi", "group"])
    seq = rng.choice([SEQ, SEQ, S2, S3])
    if kind == "field":
        return dict(kind=kind, nx=rng.randint(5, 12), nv=rng.randint(5, 9), mapping=rng.choice([SEQ, S2, S3, IF]),
                    chi=_log_int(rng, 8, 64))
    if kind == "gemm":
        return dict(kind=kind, M=_log_int(rng, 8, 1200), N=_log_int(rng, 8, 1200), K=_log_int(rng, 8, 1200),
                    precision=rng.choice(["fp64", "fp64", "fp64", "fp32", "tf32", "bf16", "tf32x3"]))
    if kind == "create":
        return dict(kind=kind, nx=rng.randint(6, 10), nv=rng.randint(6, 10), mapping=rng.choice([SEQ, S2, S3, IF]),
                    chi=_log_int(rng, 12, 64))
    if kind == "stage":
        inter = rng.random() < 0.3
        return dict(kind=kind, nx=rng.randint(5, 7 if inter else 9), nv=rng.randint(5, 7 if inter else 9),
                    mapping=IF if inter else seq, chi=_log_int(rng, 8, 32 if inter else 64))
    if kind == "run":
        return dict(kind=kind, nx=rng.randint(5, 7), nv=rng.randint(5, 7), mapping=seq, chi=_log_int(rng, 8, 32),
                    steps=rng.randint(1, 3), modes=rng.randint(3, 12))
    if kind == "step":
        inter = rng.random() < 0.2
        return dict(kind=kind, nx=rng.randint(6, 7 if inter else 10), nv=rng.randint(6, 7 if inter else 10),
                    mapping=IF if inter else seq, chi=_log_int(rng, 12, 32 if inter else 96),
                    streams=rng.choice([0, 0, 2]), modes=rng.choice([16, 32, 48]))
    if kind == "multi":
        return dict(kind=kind, nx=rng.randint(6, 9), nv=rng.randint(6, 9), mapping=seq, chi=_log_int(rng, 16, 64))
    return dict(kind="group", members=rng.randint(4, 24), low=rng.randint(5, 6), high=rng.randint(7, 8),
                chi=_log_int(rng, 12, 32))


# -------------------------------------------------------------------- the inputs
def _layout(nx, nv, mapping):
    return inputs.Layout(nx, nv, 0.0, 10 * math.pi, -8.0, 8.0, mapping)


def _dt(lay):
    """The largest stable step of the workloads: max |v| dt / dx = 0.6."""
    return 0.6 * ((lay.xmax - lay.xmin) / lay.Nx) / max(abs(lay.vmin), abs(lay.vmax))


def _state(lay, modes, seed, beams, vth, k, eps, device):
    """h(v) [1 + eps sum_m a_m cos(m k x + phi_m) psi_m(v)]: seeded broadband perturbation of
    Hermite-Gauss shapes around the beams, the state of the saturated phase."""
    rng = np.random.Generator(np.random.PCG64(seed))
    x, v = lay.x(), lay.v()
    h = sum(inputs.maxwellian(v, vth, u) for u in beams) / len(beams)
    a = rng.uniform(0.3, 1.0, size=modes) / np.arange(1, modes + 1) ** 0.5
    phi = rng.uniform(0, 2 * math.pi, size=modes)
    centre = rng.choice(np.asarray(beams, dtype=float), size=modes)
    order = rng.integers(0, 4, size=modes)
    width = rng.uniform(0.6, 1.4, size=modes) * vth
    left, right = [np.ones(lay.Nx)], [h]
    for m in range(modes):
        s = (v - centre[m]) / width[m]
        psi = np.polynomial.hermite.hermval(s, [0] * order[m] + [1]) * np.exp(-s * s / 2)
        psi = psi / np.max(np.abs(psi))
        left.append(eps * a[m] * np.cos((m + 1) * k * x + phi[m]))
        right.append(h * psi)
    ta = torch.from_numpy(np.stack(left, 1)).to(device)
    tb = torch.from_numpy(np.stack(right, 0)).to(device)
    return (ta @ tb).contiguous()


def _two_stream(lay, modes, seed, device):
    return _state(lay, modes, seed, (-3.0, 3.0), 1.0, 0.2, 0.05, device)


SPECIES = [(-1.0, 1.0, 0.007, 10.0, 1.0), (1.0, 25.0, 0.0014, 0.0, 0.2)]  # q, m, collision rate, drift, thermal speed


def _species(case, seed, device):
    lays = inputs.buneman_layouts(case["nx"], case["nv"], case["nv"], mapping=case["mapping"])
    fs = [_state(lay, MODES, 2 * seed + s, (u,), vth, 0.1, amp, device)
          for s, (lay, u, vth, amp) in enumerate(zip(lays, (10.0, 0.0), (1.0, 0.2), (0.05, 0.01)))]
    return lays, fs, _dt(lays[0])


def _members(case):
    """(layout, chi) of every simulation of a group: sizes between low and high bits, sequential
    orderings, with a small interleaved grid among each five."""
    out = []
    for i in range(case["members"]):
        if i % 5 == 4:
            out.append((_layout(case["low"], case["low"], IF), max(8, case["chi"] // 2)))
            continue
        span = case["high"] - case["low"] + 1
        nx, nv = case["low"] + i % span, case["low"] + (i // 2) % span
        out.append((_layout(nx, nv, (SEQ, S3, SEQ, S2)[i % 4]), max(8, case["chi"] - 4 * (i % 3))))
    return out


def _gemm_operands(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    M, N, K = case["M"], case["N"], case["K"]
    # an upper-graded left factor (rows falling over six decades, as R has) and a core
    A = rng.standard_normal((M, K)) * np.logspace(0, -6, M)[:, None]
    return A, rng.standard_normal((K, N)) / math.sqrt(K)


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    st = dict(kind=kind, ctx=ctx, case=case)
    if kind == "gemm":
        st["A"], st["B"] = (torch.from_numpy(t).cuda() for t in _gemm_operands(case, seed))
        st["precision"] = vpmps.PRECISIONS[case["precision"]]
        return st
    if kind == "multi":
        lays, fs, dt = _species(case, seed, "cuda")
        ms = [ctx.mps_from_grid(lay, f, case["chi"], TOL) for lay, f in zip(lays, fs)]
        st.update(lays=lays, sim=ctx.multi(lays, SPECIES, ms, dt, case["chi"]))
        return st
    if kind == "group":
        grp, sims = ctx.group(case["members"]), []
        for i, (lay, chi) in enumerate(_members(case)):
            m = ctx.mps_from_grid(lay, _two_stream(lay, MODES // 2, 100 * seed + i, "cuda"), chi, TOL)
            sims.append(ctx.sim(lay, m, _dt(lay), chi, streams=1))
            grp.add(sims[-1])
        st.update(group=grp, sims=sims)
        return st
    lay = _layout(case["nx"], case["nv"], case["mapping"])
    f = _two_stream(lay, case.get("modes", MODES), seed, "cuda")
    st["lay"] = lay
    if kind == "create":
        st["f"] = f
    elif kind == "run":
        st["f"] = f.cpu().numpy()
    else:
        st["f"] = m = ctx.mps_from_grid(lay, f, case["chi"], TOL)
        if kind == "stage":
            E = _field(f.cpu().numpy().sum(1) * _dv(lay), _dx(lay))[0]
            st.update(L=ctx.mpo_vlasov(lay, E, TOL), Lf=ctx.empty_mps(), out=ctx.empty_mps())
        elif kind == "step":
            st["sim"] = ctx.sim(lay, m, _dt(lay), case["chi"], streams=case["streams"])
    return st


# ---------------------------------------------------------------------- one pass
def _records(recs):
    return {k: [r[k] for r in recs] for k in ("t", "field_energy", "mass", "max_bond")}


def run(st):
    kind, ctx, case = st["kind"], st["ctx"], st["case"]
    if kind == "field":
        lay = st["lay"]
        rho = ctx.density(lay, st["f"])
        E, energy = ctx.poisson(rho, lay.nx, _dx(lay))
        return {"rho": rho, "E": E, "energy": energy}
    if kind == "gemm":
        return ctx.gemm(st["A"], st["B"], precision=st["precision"])
    if kind == "create":
        m = ctx.mps_from_grid(st["lay"], st["f"], case["chi"], TOL)
        return m.to_grid(st["lay"])
    if kind == "stage":
        ctx.apply_mpo(st["L"], st["f"], st["Lf"])
        ctx.axpby(1.0, st["f"], _dt(st["lay"]), st["Lf"], st["out"])
        ctx.compress(st["out"], case["chi"], TOL)
        return st["out"].to_grid(st["lay"])
    if kind == "run":
        f, recs = ctx.run(st["lay"], st["f"], _dt(st["lay"]), case["steps"], case["chi"])
        return {"f": f, **_records(recs)}
    if kind == "step":
        recs = st["sim"].step(1)
        return {"f": st["sim"].state().to_grid(st["lay"]), **_records(recs)}
    if kind == "multi":
        rec = st["sim"].step(1)[0]
        return {"f": [st["sim"].state(s).to_grid(lay) for s, lay in enumerate(st["lays"])],
                **{k: rec[k] for k in ("t", "field_energy", "mass", "max_bond")}}
    recs, status = st["group"].step()
    r = {k: np.array(v) for k, v in _records(recs).items()}
    return {"f": [s.state().to_grid(s.lay) for s in st["sims"]], "status": np.array(status), **r}


# --------------------------------------------------- what a pass cannot do without
def _bonds(n, cap):
    return [min(2 ** min(k, n - k), cap) for k in range(n + 1)]


def _compress_flops(n, inner, cap):
    """QR of every site of an MPS with inner bond `inner`, then the SVD of every site at bond `cap`."""
    r, s, fl = _bonds(n, inner), _bonds(n, cap), 0.0
    for k in range(n):
        m, w = 2 * r[k], r[k + 1]
        fl += 4.0 * m * w * min(m, w)
        m, w = r[k], 2 * s[k + 1]
        fl += 6.0 * m * w * min(m, w)
    return fl


def _mps_bytes(n, cap):
    r = _bonds(n, cap)
    return 8.0 * sum(2 * r[k] * r[k + 1] for k in range(n))


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (M * K + K * N + M * N), "flops": 2.0 * M * N * K}
    if kind == "group":
        w = [work(dict(kind="step", nx=lay.nx, nv=lay.nv, mapping=lay.mapping, chi=chi)) for lay, chi in _members(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "multi":
        w = work(dict(case, kind="step"))
        return {k: 2 * v for k, v in w.items()}
    n, chi, grid = case["nx"] + case["nv"], case["chi"], 8.0 * 2 ** (case["nx"] + case["nv"])
    if kind == "field":
        return {"bytes": _mps_bytes(n, chi) + 16.0 * 2 ** case["nx"], "flops": 2.0 * chi * 2 ** case["nx"] + 4.0 * case["nv"] * chi * chi}
    if kind == "create":
        # the unfoldings' factorisations down to the cap, then the expansion
        return {"bytes": 2 * grid, "flops": grid / 8 * 8.0 * chi}
    one = _compress_flops(n, 4 * chi, chi)
    if kind == "stage":
        return {"bytes": 2 * _mps_bytes(n, chi) + grid, "flops": one}
    steps = case.get("steps", 1)  # seven compressions a step
    return {"bytes": 2 * _mps_bytes(n, chi) + grid * (2 if kind == "run" else 1), "flops": 7.0 * steps * one}


# ---------------------------------------------------------- the same, on the full grid
def _dx(lay):
    return (lay.xmax - lay.xmin) / lay.Nx


def _dv(lay):
    return (lay.vmax - lay.vmin) / (lay.Nv - 1)


def _field(rho, dx):
    """E of the periodic second-order Poisson problem and its energy."""
    s = np.concatenate([[0.0], np.cumsum(dx * dx * (rho[1:] - rho.mean()))])
    d = s - s.mean()
    E = -(d + np.roll(d, 1)) / (2 * dx)
    return E, 0.5 * float((E * E).sum()) * dx


def _rhs(f, lay, E, nu=0.0, u=0.0, vth=1.0):
    dx, dv, v = _dx(lay), _dv(lay), lay.v()
    back = (1.5 * f - 2.0 * np.roll(f, 1, 0) + 0.5 * np.roll(f, 2, 0)) / dx
    fore = (-1.5 * f + 2.0 * np.roll(f, -1, 0) - 0.5 * np.roll(f, -2, 0)) / dx
    out = -np.where(v > 0, v, 0.0) * back - np.where(v > 0, 0.0, v) * fore

    def dc(g):
        o = np.zeros_like(g)
        o[:, 1:-1] = (g[:, 2:] - g[:, :-2]) / (2 * dv)
        return o

    out += E[:, None] * dc(f)
    if nu:
        g = np.empty_like(f)
        g[:, 1:-1] = (f[:, 2:] - 2 * f[:, 1:-1] + f[:, :-2]) / (dv * dv)
        g[:, 0] = 2 * (f[:, 1] - f[:, 0]) / (dv * dv)
        g[:, -1] = 2 * (f[:, -2] - f[:, -1]) / (dv * dv)
        out += nu * (dc((v - u) * f) + vth * vth * g)
    return out


def _rk4(fs, lays, species, dt):
    """One step of every species on the common field: new f's, field energy and masses of the old ones."""
    dx = _dx(lays[0])

    def rhs(gs):
        rhos = [g.sum(1) * _dv(lay) for g, lay in zip(gs, lays)]
        E, we = _field(-sum(sp[0] * r for sp, r in zip(species, rhos)), dx)
        return [_rhs(g, lay, -sp[0] / sp[1] * E, *sp[2:]) for g, lay, sp in zip(gs, lays, species)], we, rhos

    def ahead(a, ks):
        return [f + a * dt * k for f, k in zip(fs, ks)]

    k1, we, rhos = rhs(fs)
    k2 = rhs(ahead(0.5, k1))[0]
    k3 = rhs(ahead(0.5, k2))[0]
    k4 = rhs(ahead(1.0, k3))[0]
    new = [f + dt / 6 * (a + 2 * b + 2 * c + d) for f, a, b, c, d in zip(fs, k1, k2, k3, k4)]
    return new, we, [float(r.sum()) * dx for r in rhos]


def _axes(lay):
    """Site order of the bits of f[ix, iv] reshaped to 2 x 2 x ..., x bits first."""
    xs, vs = list(range(lay.nx)), list(range(lay.nx, lay.nx + lay.nv))
    if lay.mapping == S2:
        return xs[::-1] + vs
    if lay.mapping == S3:
        return xs + vs[::-1]
    if lay.mapping == IF:
        return [a for b in range(max(lay.nx, lay.nv)) for a in xs[b:b + 1] + vs[b:b + 1]]
    return xs + vs


def _truncate(f, lay, chi):
    """(f after the right-to-left sweep of truncated SVDs, its largest bond)."""
    n, axes = lay.nx + lay.nv, _axes(lay)
    left, right, r, most = np.ascontiguousarray(f.reshape((2,) * n).transpose(axes)).reshape(-1), [], 1, 1
    for k in range(n - 1, 0, -1):
        m = left.reshape(-1, 2 * r)
        q = None
        if m.shape[0] > 4 * m.shape[1]:
            q, m = np.linalg.qr(m)
        u, s, vt = np.linalg.svd(m, full_matrices=False)
        tail = np.sqrt(np.cumsum((s * s)[::-1])[::-1]) / np.linalg.norm(s)
        small = np.nonzero(tail[1:] <= TOL)[0]
        keep = max(1, min(chi, small[0] + 1 if small.size else s.size))
        while 1 < keep < s.size and s[keep - 1] - s[keep] <= 1e-5 * s[keep - 1]:
            keep -= 1
        us = u[:, :keep] * s[:keep]
        left = (us if q is None else q @ us).reshape(-1)
        right.append(vt[:keep].reshape(keep, 2, r))
        r, most = keep, max(most, keep)
    out = left.reshape(2, r)
    for c in right[::-1]:
        out = (out @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    return np.ascontiguousarray(out.reshape((2,) * n).transpose(np.argsort(axes))).reshape(lay.Nx, lay.Nv), most


ELECTRONS = [(-1.0, 1.0)]


def _steps(f, lay, chi, steps):
    dt, recs = _dt(lay), dict(t=[], field_energy=[], mass=[], max_bond=[])
    for n in range(steps):
        (f,), we, mass = _rk4([f], [lay], ELECTRONS, dt)
        f, most = _truncate(f, lay, chi)
        for k, v in (("t", n * dt), ("field_energy", we), ("mass", mass[0]), ("max_bond", most)):
            recs[k].append(v)
    return {"f": f, **recs}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B = _gemm_operands(case, seed)
        return A @ B
    if kind == "multi":
        lays, fs, dt = _species(case, seed, "cpu")
        fs = [_truncate(f.numpy(), lay, case["chi"])[0] for f, lay in zip(fs, lays)]
        fs, we, mass = _rk4(fs, lays, SPECIES, dt)
        cut = [_truncate(f, lay, case["chi"]) for f, lay in zip(fs, lays)]
        return {"f": [c[0] for c in cut], "t": 0.0, "field_energy": we, "mass": mass, "max_bond": [c[1] for c in cut]}
    if kind == "group":
        got = []
        for i, (lay, chi) in enumerate(_members(case)):
            f = _two_stream(lay, MODES // 2, 100 * seed + i, "cpu").numpy()
            got.append(_steps(_truncate(f, lay, chi)[0], lay, chi, 1))
        return {"f": [g["f"] for g in got], "status": np.zeros(len(got), dtype=np.int64),
                **{k: np.array([g[k][0] for g in got]) for k in ("t", "field_energy", "mass", "max_bond")}}
    lay = _layout(case["nx"], case["nv"], case["mapping"])
    f = _two_stream(lay, case.get("modes", MODES), seed, "cpu").numpy()
    cut = _truncate(f, lay, case["chi"])[0]
    if kind == "create":
        return cut
    if kind == "field":
        rho = cut.sum(1) * _dv(lay)
        E, we = _field(rho, _dx(lay))
        return {"rho": rho, "E": E, "energy": we}
    if kind == "stage":
        E = _field(f.sum(1) * _dv(lay), _dx(lay))[0]
        return _truncate(cut + _dt(lay) * _rhs(cut, lay, E), lay, case["chi"])[0]
    return _steps(cut, lay, case["chi"], case.get("steps", 1))
