"""What a user of this framework has it do, as cases that can be timed.

Every case goes through the public binding (``paper_2007_14401_gb300.gcb``):
a case is a dict of plain values, ``prepare`` makes what a program has in hand
before the call (grid, particle state, parameters, workspace), ``run`` makes
one pass and returns the updated state (and current or gradients), ``work``
counts what a pass cannot do without and ``exact`` computes the same pass in
64 bits with plain torch, from the method's equations.

Families (``kind``):
  flat     the flat-space push; sort_every > 0: one sort cycle per pass, the
           way long runs are driven, outputs handed back in particle-id order
  graph    the flat-space push captured by gcb.StepGraph and replayed
  pic      PiC steps: current zeroed, push with deposition
  adjoint  gcb.ModePush forward and backward
  kerr     the covariant Kerr-Schild push
Inputs follow the generators of ``inputs.py`` (Harris sheet, reconnection
field with Fourier modes, 3D kinked sheet, Wald field), drawn on the GPU.
"""
import functools
import math

import numpy as np
import torch

from paper_2007_14401_gb300 import gcb, inputs

DEV = "cuda"
F64 = torch.float64


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _flat(name, field, n, grid, precision, steps, sort_every=0, fuse=0, option="plain",
          pos="pair", kind="flat"):
    nx, ny, nz = (tuple(grid) + (1,))[:3]
    c = dict(kind=kind, field=field, n=int(n), nx=int(nx), ny=int(ny), nz=int(nz),
             precision=precision, steps=int(steps), sort_every=int(sort_every), fuse=int(fuse),
             option=option, pos=pos)
    return dict(c, name=name) if name else c


def _adjoint(name, n, grid, precision, steps, ckpt, modes, iters):
    c = dict(kind="adjoint", field="recon", n=int(n), nx=int(grid[0]), ny=int(grid[1]), nz=1,
             precision=precision, steps=int(steps), ckpt=int(ckpt), modes=int(modes),
             iters=int(iters))
    return dict(c, name=name) if name else c


def _kerr(name, n, grid, records, basis, steps):
    c = dict(kind="kerr", n=int(n), nx=int(grid[0]), ny=int(grid[1]), records=records,
             basis=basis, steps=int(steps))
    return dict(c, name=name) if name else c


def listed():
    return [
        # the correctness workload, one call a step: latency and launches count
        _flat("harris_fp64_step", "harris", 16384, (128, 128), "fp64", 1),
        # the same driven the way the binding recommends for small problems
        _flat("harris_fp64_graph", "harris", 16384, (128, 128), "fp64", 16, kind="graph"),
        # an ordinary mixed-precision run: 8 steps and the sort that starts them
        _flat("recon_mixed_1m", "recon", 1 << 20, (512, 256), "mixed", 8, sort_every=8),
        # the benchmark's workload at full size
        _flat("recon_mixed_16m", "recon", 1 << 24, (2048, 1024), "mixed", 8, sort_every=8),
        # 3D, gradients from the shape functions, both branches populated
        _flat("sheet3d_mixed_16m", "sheet", 1 << 24, (256, 256, 256), "mixed", 8, sort_every=8),
        # the FP64 path on gradient records: reference runs beside a mixed one
        _flat("recon_fp64_1m", "recon", 1 << 20, (512, 256), "fp64", 1),
        # the FP64 path in 3D on an odd grid with a ragged particle count
        _flat("sheet3d_fp64_odd", "sheet", 300007, (129, 127, 96), "fp64", 1),
        # test-particle mode (several steps per launch), ragged count, odd grid
        _flat("recon_mixed_fused_odd", "recon", 3000017, (1021, 509), "mixed", 8, sort_every=8,
              fuse=8),
        # PiC steps with the current deposited
        _flat("recon_pic_4m", "recon", 1 << 22, (1024, 512), "mixed", 8, sort_every=8, kind="pic"),
        # training: gradients of a multi-step push, forward and backward
        _adjoint("recon_adjoint_256k", 1 << 18, (512, 256), "mixed", 16, 8, 64, 6),
        # black-hole runs: local-frame kicks on FP32 records ...
        _kerr("kerr_1m", 1 << 20, (512, 512), "f32", "tetrad", 1),
        # ... and global-basis kicks on FP64 records, ragged count
        _kerr("kerr_global_odd", 100003, (301, 257), "f64", "global", 1),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flat2", "flat2", "flat3", "fp64_2", "fp64_3", "harris", "graph", "pic2",
                       "pic3", "adjoint", "kerr", "kerr"])
    g2 = (_logint(rng, 256, 2048), _logint(rng, 128, 1024))
    g3 = (_logint(rng, 96, 256), _logint(rng, 96, 256), _logint(rng, 96, 256))
    sort = rng.choice([4, 8, 8, 8])
    if kind == "flat2":
        opt = rng.choice(["plain", "plain", "plain", "exact_frame", "mirror"])
        fuse = rng.choice([0, 0, 4]) if opt == "plain" else 0
        return _flat(None, "recon", _logint(rng, 4000, 1 << 24), g2, "mixed", 8, sort, fuse, opt,
                     rng.choice(["pair", "pair", "f64"]) if opt != "exact_frame" else "pair")
    if kind == "flat3":
        return _flat(None, "sheet", _logint(rng, 4000, 1 << 23), g3, "mixed", 8, sort,
                     rng.choice([0, 0, 4]))
    if kind == "fp64_2":
        opt = rng.choice(["plain", "plain", "exact_frame", "phase", "mirror"])
        return _flat(None, "recon", _logint(rng, 4000, 1 << 20), g2, "fp64", rng.choice([1, 2]),
                     option=opt)
    if kind == "fp64_3":
        return _flat(None, "sheet", _logint(rng, 4000, 1 << 20), g3, "fp64", rng.choice([1, 2]))
    if kind in ("harris", "graph"):
        n = _logint(rng, 1000, 200000)
        g = (_logint(rng, 64, 256), _logint(rng, 64, 256))
        if kind == "graph":
            return _flat(None, "harris", n, g, "fp64", rng.choice([4, 16]), kind="graph")
        return _flat(None, "harris", n, g, "fp64", 1)
    if kind == "pic2":
        mixed = rng.random() < 0.8
        return _flat(None, "recon", _logint(rng, 4000, (1 << 22) if mixed else (1 << 18)), g2,
                     "mixed" if mixed else "fp64", 4, sort, kind="pic")
    if kind == "pic3":
        return _flat(None, "sheet", _logint(rng, 4000, 1 << 22), g3, "mixed", 4, sort, kind="pic")
    if kind == "adjoint":
        f64 = rng.random() < 0.3
        g = (_logint(rng, 128, 512), _logint(rng, 64, 256))
        return _adjoint(None, _logint(rng, 2000, (1 << 15) if f64 else (1 << 18)), g,
                        "fp64" if f64 else "mixed", rng.choice([4, 8, 12]), rng.choice([4, 8]),
                        _logint(rng, 4, 64), rng.choice([4, 6]))
    return _kerr(None, _logint(rng, 3000, 1 << 20), (_logint(rng, 128, 512), _logint(rng, 128, 512)),
                 rng.choice(["f32", "f64"]), rng.choice(["tetrad", "global"]), rng.choice([1, 2]))


# --------------------------------------------------------------------------
# inputs: fields and particles, float64 on the GPU, from the seed alone
# --------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uni(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _isotropic(g, mag):
    mu, ph = _uni(g, mag.numel(), lo=-1.0), _uni(g, mag.numel(), hi=2 * math.pi)
    s = torch.sqrt(1.0 - mu * mu)
    return torch.stack([s * torch.cos(ph), s * torch.sin(ph), mu]) * mag


@functools.lru_cache(maxsize=8)
def _mj_table(theta):
    """Kinetic energies and their distribution function (host: a scan on the
    GPU would round differently from run to run)."""
    e = np.linspace(0.0, 60.0 * theta + 1.0, 1 << 17)
    f = np.sqrt(e * (e + 2.0)) * (1.0 + e) * np.exp(-e / theta)
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (f[1:] + f[:-1]))])
    return torch.from_numpy(e).to(DEV), torch.from_numpy(cdf / cdf[-1]).to(DEV)


def _maxwell_juttner(g, n, theta):
    """Isotropic momenta of temperature theta, by inverse transform."""
    e, cdf = _mj_table(theta)
    U = _uni(g, n)
    k = torch.searchsorted(cdf, U).clamp_(1, e.numel() - 1)
    w = (U - cdf[k - 1]) / (cdf[k] - cdf[k - 1]).clamp_min(1e-300)
    ek = e[k - 1] + w * (e[k] - e[k - 1])
    return _isotropic(g, torch.sqrt(ek * (ek + 2.0)))


def _power_law(g, n, gmax):
    gam = 1.0 / (1.0 - _uni(g, n) * (1.0 - 1.0 / gmax))
    return _isotropic(g, torch.sqrt((gam * gam - 1.0).clamp_min(0.0)))


def _central(B):
    """Central differences d_i B_j (i over x, y), unit spacing."""
    return [(torch.roll(b, -1, 1 - i) - torch.roll(b, 1, 1 - i)) / 2.0 for i in range(2) for b in B]


def _mode_numbers(g, modes):
    def num():
        k = torch.randint(1, 17, (modes,), generator=g, device=DEV)
        return (k * (2 * torch.randint(0, 2, (modes,), generator=g, device=DEV) - 1)).tolist()
    return list(zip(num(), num(), _uni(g, modes, hi=2 * math.pi).tolist()))


GUIDE = 0.3      # B_z (without one the field has null points, where trajectories part)


def _recon_base(nx, ny):
    X = torch.arange(nx, device=DEV, dtype=F64)[None, :].expand(ny, nx)
    Y = (torch.arange(ny, device=DEV, dtype=F64) - 0.5 * ny)[:, None].expand(ny, nx)
    d = 8.0 if ny >= 256 else ny / 32.0
    kx, ky, psi0 = 2 * math.pi / nx, math.pi / ny, 0.1
    Bx = torch.tanh((Y + ny / 4) / d) - torch.tanh((Y - ny / 4) / d) - 1.0
    Bx = Bx + psi0 * ky * torch.cos(kx * X) * torch.sin(ky * Y)
    By = -psi0 * kx * torch.sin(kx * X) * torch.cos(ky * Y)
    return X, Y, Bx, By, 0.1 * torch.sin(4 * math.pi * Y / ny)


def _mode(X, Y, v, m):
    """Bx, By of one Fourier mode of unit amplitude."""
    ny, nx = X.shape
    kx, ky = 2 * math.pi * m[0] / nx, 2 * math.pi * m[1] / ny
    s = torch.sin(kx * X + ky * Y + m[2]) / math.hypot(kx, ky)
    return ky * s, -kx * s


def _recon_fields(nx, ny, g):
    X, Y, Bx, By, v = _recon_base(nx, ny)
    for m in _mode_numbers(g, 64):
        bx, by = _mode(X, Y, v, m)
        Bx, By = Bx + 0.02 * bx, By + 0.02 * by
    Z = torch.zeros_like(Bx)
    B = [Bx, By, Z + GUIDE]
    return dict(E=[-v * B[2], Z, v * Bx], B=B, dB=_central(B), dx=(1.0, 1.0))


def _harris_fields(nx, ny):
    Y = (torch.arange(ny, device=DEV, dtype=F64) - 0.5 * ny)[:, None].expand(ny, nx)
    Z = torch.zeros((ny, nx), device=DEV, dtype=F64)
    return dict(E=[Z, Z, Z + 0.05], B=[torch.tanh(Y / 4.0), Z, Z + 0.1], dB=None, dx=(1.0, 1.0))


def _sheet_fields(nx, ny, nz):
    z = torch.arange(nz, device=DEV, dtype=F64)[:, None, None]
    y = (torch.arange(ny, device=DEV, dtype=F64) - 0.5 * ny)[None, :, None]
    Z = torch.zeros((nz, ny, nx), device=DEV, dtype=F64)
    Bx = Z + torch.tanh((y - 0.05 * ny * torch.sin(2 * math.pi * z / nz)) / 6.0)
    return dict(E=[Z, Z + 0.1, Z], B=[Bx, Z, Z + 0.3], dB=None, dx=(1.0, 1.0, 1.0))


def _flat_inputs(c, seed):
    """(fields, state, params): float64 tensors, the state rounded to what the
    case's precision holds."""
    g = _gen(seed)
    n, dims = c["n"], ((c["nx"], c["ny"]) if c["nz"] == 1 else (c["nx"], c["ny"], c["nz"]))
    p = dict(c=1.0, f_rho=0.4, f_E=1.0, dl=1.0, curvature=1, mu_mode=0, gca_max_iter=16,
             gca_tol=1e-7, dt=0.45, grad_mode=0)
    sp = torch.arange(n, device=DEV) % 2
    if c["field"] == "harris":
        f = _harris_fields(*dims)
        u = _maxwell_juttner(g, n, 0.1)
        p.update(dt=0.25, qm=(-1.0, -10.0, -100.0, -1000.0))
        sp = torch.arange(n, device=DEV) * 4 // n
    elif c["field"] == "recon":
        f = _recon_fields(*dims, g)
        u = _maxwell_juttner(g, n, 1.0)
        # Omega_C dt up to 100: rounding of E.b is amplified by q/m, so that at
        # 1e5 float32 results are only determined to 1e-4
        q = 1e2 / (p["dt"] * float(torch.sqrt(sum(b * b for b in f["B"])).max()))
        p.update(qm=(-q, q), grad_mode=1)
    else:
        f = _sheet_fields(*dims)
        nth = int(round(0.7 * n))
        u = torch.cat([_maxwell_juttner(g, nth, 0.3), _power_law(g, n - nth, 1e4)], 1)
        p.update(qm=(-20.0, 20.0))
    x = torch.stack([_uni(g, n, hi=float(L)) for L in dims])
    if c["field"] == "sheet":      # thermal upstream, power law inside the sheet
        ny, nz = dims[1], dims[2]
        off = torch.where(torch.arange(n, device=DEV) < nth, 12.0 + x[1] / ny * (ny - 24.0),
                          6.0 * (2.0 * x[1] / ny - 1.0))
        x[1] = torch.remainder(0.5 * ny + 0.05 * ny * torch.sin(2 * math.pi * x[2] / nz) + off, ny)
    if c.get("sort_every", 0) or c["kind"] == "adjoint":   # a run under way is near cell order
        key = torch.zeros(n, device=DEV, dtype=torch.int64)
        for d in reversed(range(len(dims))):
            key = key * dims[d] + x[d].floor().long().clamp_(0, dims[d] - 1)
        o = torch.argsort(key, stable=True)
        x, u, sp = x[:, o], u[:, o], sp[o]
    dxp = p["dt"] * u[:len(dims)] / torch.sqrt(1.0 + (u * u).sum(0))
    if c["precision"] == "mixed":
        u, dxp = u.float().double(), dxp.float().double()
        if c.get("pos", "pair") == "pair":
            hi = x.float().double()
            x = hi + (x - hi).float().double()
    st = dict(x=x.contiguous(), u=u.contiguous(), dxp=dxp.contiguous(),
              flags=(sp << gcb.SPECIES_SHIFT).to(torch.uint8))
    return f, st, p


def _grid(f, dtype):
    host = {k: None if f[k] is None else [t.cpu().numpy() for t in f[k]] for k in ("E", "B", "dB")}
    return gcb.Grid(dict(host, dx=f["dx"]), dtype=dtype)


OPTIONS = dict(plain={}, exact_frame=dict(drift_frame=1), phase=dict(gyro_phase=1),
               mirror=dict(mirror=1))


def _prepare_flat(c, seed):
    f, st, p = _flat_inputs(c, seed)
    fp64 = c["precision"] == "fp64"
    grid = _grid(f, "f64" if fp64 else "f32")
    nd = 2 if c["nz"] == 1 else 3
    ds = gcb.State(c["n"], nd, c["precision"], c["pos"], with_pid=c["sort_every"] > 0)
    ds.set_tensors(st["x"], st["u"], st["dxp"], st["flags"])
    gp = gcb.make_params(p, sort_every=c["sort_every"], sort_tile=(1,) * nd, fuse_steps=c["fuse"],
                         **OPTIONS[c["option"]])
    s = dict(case=c, state=ds, grid=grid, gp=gp, ws=gcb.Workspace(ds, grid, gp))
    if c["sort_every"]:
        s["ids"] = torch.arange(c["n"], device=DEV)
    if c["kind"] == "pic":
        s["cur"] = gcb.Current(grid, (-1.0, 1.0), c["precision"])
    if c["kind"] == "graph":
        # the first call sizes the kernels; then back to the initial particles
        gcb.push(ds, grid, gp, 1, workspace=s["ws"], stats=False)
        ds.set_tensors(st["x"], st["u"], st["dxp"], st["flags"])
        s["graph"] = gcb.StepGraph(ds, grid, gp, c["steps"], s["ws"])
    return s


def _mode_records(c, seed):
    """Base and pattern records of the mode fields (node record layout) and
    the amplitudes."""
    g = _gen(seed + 77)
    X, Y, Bx, By, v = _recon_base(c["nx"], c["ny"])

    def rec(bx, by, bz=0.0):
        Z = torch.zeros_like(bx)
        B = [bx, by, Z + bz]
        return torch.stack([-v * B[2], Z, v * bx, *B, *_central(B)], -1).reshape(-1)

    dt = F64 if c["precision"] == "fp64" else torch.float32
    base = rec(Bx, By, GUIDE).to(dt)
    pat = torch.empty((c["modes"], base.numel()), device=DEV, dtype=dt)
    for k, m in enumerate(_mode_numbers(g, c["modes"])):
        pat[k] = rec(*_mode(X, Y, v, m))
    amps = 0.02 * (1.0 + 0.2 * torch.randn(c["modes"], generator=g, device=DEV, dtype=F64))
    return base, pat, amps


def _prepare_adjoint(c, seed):
    f, st, p = _flat_inputs(c, seed)
    mixed = c["precision"] == "mixed"
    base, pat, amps = _mode_records(c, seed)
    mdt = torch.float32 if mixed else F64
    leaf = [t.requires_grad_() for t in (st["x"], st["u"].to(mdt), st["dxp"].to(mdt), amps)]
    cfg = dict(grid=_grid(f, "f32" if mixed else "f64"), base=base, pat=pat,
               params=gcb.make_params(p, gca_fixed_iters=c["iters"], sort_every=c["ckpt"],
                                      sort_tile=(1, 1)),
               n_steps=c["steps"], ckpt_every=c["ckpt"], flags=st["flags"],
               precision=c["precision"], pos_mode="pair" if mixed else "f64")
    return dict(case=c, leaf=leaf, cfg=cfg)


@functools.lru_cache(maxsize=4)
def _kerr_fields(nr, nth):
    f, _, p = inputs.kerr_wald(nr=nr, nth=nth, n_particles=16)
    return f, p


def _kerr_inputs(c, seed):
    """Electrons uniform in (log r, theta, phi), thermal in the normal frame."""
    g = _gen(seed)
    f, p = _kerr_fields(c["nx"], c["ny"])
    n = c["n"]
    r = torch.exp(_uni(g, n, lo=float(f["logr0"]), hi=math.log(float(f["r_out"]))))
    th = torch.arccos(_uni(g, n, lo=-0.98, hi=0.98))
    h = _maxwell_juttner(g, n, 1.0)
    m = _metric(f["a"], r, th, False)
    l00 = m["grr"].sqrt()
    l20 = m["grp"] / l00
    l22 = (m["gpp"] - l20 * l20).sqrt()
    u2 = h[2] / l22
    u = torch.stack([(h[0] - l20 * u2) / l00, h[1] / m["gtt"].sqrt(), u2])
    return f, p, torch.stack([r, th, _uni(g, n, hi=2 * math.pi)]), u


def _prepare_kerr(c, seed):
    f, p, x, u = _kerr_inputs(c, seed)
    grid = gcb.KsGrid(f, p["a"], p["r_in"], p["r_out"], dtype=c["records"],
                      kick_basis=gcb.KS_TETRAD if c["basis"] == "tetrad" else gcb.KS_GLOBAL)
    ds = gcb.State(c["n"], 3, "fp64")
    ds.set_tensors(x, u, torch.zeros_like(x), torch.zeros(c["n"], device=DEV, dtype=torch.uint8))
    return dict(case=c, state=ds, grid=grid, gp=gcb.make_params(p), ws=gcb.ks_workspace())


def prepare(case, seed):
    if case["kind"] == "adjoint":
        s = _prepare_adjoint(case, seed)
    elif case["kind"] == "kerr":
        s = _prepare_kerr(case, seed)
    else:
        s = _prepare_flat(case, seed)
    torch.cuda.synchronize()
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _outputs(s):
    """The state as a program reads it; after a sort, by particle id."""
    ds = s["state"]
    # mixed path: positions as float32 (x_lo refines them below their last place)
    x = ds.x if ds.precision == "fp64" else ds.x.float()
    if ds.pid is None:
        return dict(x=x, u=ds.u, dxp=ds.dxp, flags=ds.flags)
    row = torch.empty_like(ds.pid)
    row[ds.pid] = s["ids"]
    return dict(x=x[:, row], u=ds.u[:, row], dxp=ds.dxp[:, row], flags=ds.flags[row])


def run(s):
    c = s["case"]
    if c["kind"] == "adjoint":
        x, u, dxp = gcb.ModePush.apply(*s["leaf"], s["cfg"])
        # kinetic energy and mean displacement
        loss = (torch.sqrt(1.0 + (u * u).sum(0)) - 1.0).sum() + x.sum()
        gx, gu, gd, ga = torch.autograd.grad(loss, s["leaf"])
        # in the precision they are computed in (the momenta's)
        return dict(x=x.detach().to(u.dtype), u=u.detach(), dxp=dxp.detach(), gx=gx.to(u.dtype), gu=gu,
                    gdxp=gd, gamps=ga.to(u.dtype))
    if c["kind"] == "kerr":
        ds = s["state"]
        gcb.push_ks(ds, s["grid"], s["gp"], c["steps"], workspace=s["ws"], stats=False)
        return dict(x=ds.x, u=ds.u, flags=ds.flags)
    if c["kind"] == "graph":
        s["graph"].replay()
        return _outputs(s)
    if c["kind"] == "pic":
        for k in range(c["steps"]):
            s["cur"].zero()
            s["gp"].step_index = k
            gcb.push(s["state"], s["grid"], s["gp"], 1, workspace=s["ws"], stats=False,
                     current=s["cur"])
        return dict(_outputs(s), J=s["cur"].J)
    gcb.push(s["state"], s["grid"], s["gp"], c["steps"], workspace=s["ws"], stats=False)
    return _outputs(s)


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
# floating-point operations of one particle-step: gathers (2 per node and
# component, ~5 of them), local frames and velocities at each
STEP_FLOPS = {2: 1400.0, 3: 2200.0}
KERR_FLOPS = 1700.0
ADJOINT_FLOPS = 4.0      # reverse step (replay and transpose) over a forward step


def work(c):
    n, nodes = c["n"], c["nx"] * c["ny"] * c.get("nz", 1)
    if c["kind"] == "kerr":
        return dict(bytes=2 * 49 * n + nodes * 6 * (4 if c["records"] == "f32" else 8),
                    flops=KERR_FLOPS * n * c["steps"])
    nd = 2 if c["nz"] == 1 else 3
    e = 8 if c["precision"] == "fp64" else 4
    comps = 12 if c["field"] == "recon" else 6
    state = 8 * nd + e * (3 + nd) + 1
    if c["kind"] == "adjoint":
        # inputs, outputs and gradients once each; mode patterns read by the
        # combination and by the projection
        b = n * (3 * 8 * nd + 3 * e * (3 + nd) + 1) + 2 * nodes * 12 * e * c["modes"]
        return dict(bytes=b, flops=n * c["steps"] * STEP_FLOPS[2] * (1.0 + ADJOINT_FLOPS))
    b = 2 * state * n + nodes * comps * e
    if c["kind"] == "pic":       # the fields may change between PiC steps: state once a step
        b = c["steps"] * (b + 3 * nodes * e)
    return dict(bytes=b, flops=n * c["steps"] * STEP_FLOPS[nd])


# --------------------------------------------------------------------------
# the same pass in 64 bits, from the method's equations
# --------------------------------------------------------------------------
CHUNK = 1 << 20


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2],
                        a[0] * b[1] - a[1] * b[0]])


def _gather(rec, dims, x):
    """E, B (3, m) and d_i B_j (nd lists of (3, m)) at x; rec (nodes, 6 | 12),
    unit spacing, periodic; six components: gradients of the shape functions."""
    nd = len(dims)
    fl = torch.floor(x.detach())
    t = x - fl
    i0 = [torch.remainder(fl[d].long(), dims[d]) for d in range(nd)]
    i1 = [torch.remainder(i0[d] + 1, dims[d]) for d in range(nd)]
    out, dB = 0.0, [0.0] * nd
    for o in range(1 << nd):
        hi = [(o >> d) & 1 for d in range(nd)]
        w = [t[d] if hi[d] else 1.0 - t[d] for d in range(nd)]
        idx = 0
        for d in reversed(range(nd)):
            idx = idx * dims[d] + (i1[d] if hi[d] else i0[d])
        v = rec.index_select(0, idx).t()
        W = w[0]
        for d in range(1, nd):
            W = W * w[d]
        out = out + W * v
        if rec.shape[1] == 6:
            for i in range(nd):
                gw = 1.0 if hi[i] else -1.0
                for d in range(nd):
                    if d != i:
                        gw = gw * w[d]
                dB[i] = dB[i] + gw * v[3:6]
    if rec.shape[1] == 12:
        dB = [out[6:9], out[9:12]]
    return out[0:3], out[3:6], dB


def _frame(F, opt):
    E, B, dB = F
    B2 = _dot(B, B)
    Bm = torch.sqrt(B2)
    bl = B / Bm
    f = dict(Bm=Bm)
    if opt == "exact_frame":
        E2, EB = _dot(E, E), _dot(E, B)
        S, D = E2 + B2, B2 - E2
        s = torch.sqrt(D * D + 4.0 * EB * EB) / S
        vE = 2.0 * _cross(E, B) / (S * (1.0 + s))
        Bp = torch.sqrt(0.5 * (S * s + D))
        ep = E - EB / B2 * B
        psi = 2.0 * EB / Bp * B2 / (Bp * S * (1.0 + s))
        eta = 1.0 / (Bm * torch.sqrt(psi * psi * _dot(ep, ep) / B2 + 1.0))
        b = eta * psi * ep + eta * B
    else:
        b, vE = bl, _cross(E, B) / B2
    f["kap"] = 1.0 / torch.sqrt(1.0 - _dot(vE, vE))
    w = sum(b[i] * dB[i] for i in range(len(dB)))
    y = sum(vE[i] * dB[i] for i in range(len(dB)))
    f.update(b=b, vE=vE, Epar=_dot(E, b), bgb=(w - bl * _dot(bl, w)) / Bm,
             vgb=(y - bl * _dot(bl, y)) / Bm)
    if opt == "mirror":
        g = [_dot(bl, d) for d in dB]
        f["gB"] = torch.stack(g + [torch.zeros_like(Bm)] * (3 - len(g)))
    return f


def _gamma(f, up, mu):
    return f["kap"] * torch.sqrt(1.0 + up * up + 2.0 * mu * f["Bm"] * f["kap"])


def _vc(f, qm, up, G):
    return f["kap"] ** 2 / (qm * f["Bm"]) * _cross(f["b"], up * up / G * f["bgb"] + up * f["vgb"])


def _vel(f, qm, up, mu, opt):
    G = _gamma(f, up, mu)
    v = up / G * f["b"] + f["vE"] + _vc(f, qm, up, G)
    if opt == "mirror":
        v = v + f["kap"] * mu / (qm * G * f["Bm"]) * _cross(f["b"], f["gB"])
    return v


def _gca(rec, dims, x, u, dxp, qm, dt, F0, opt, iters):
    """One guiding-center step: (ok, u, displacement, z velocity).  iters > 0:
    that many fixed-point iterations; else until the change is below 1e-7."""
    nd = len(dims)
    f0 = _frame(F0, opt)
    f = _frame(_gather(rec, dims, x - 0.5 * dxp), opt)
    Gf = torch.sqrt(1.0 + _dot(u, u))
    up = _dot(u, f["b"])
    ug = u - up * f["b"] - (f["vE"] + _vc(f, qm, up, Gf)) * Gf
    uperp = torch.sqrt(_dot(ug, ug))
    bpg = ug / uperp
    mu = uperp * uperp / (2.0 * f["Bm"] * f["kap"])
    a, gg = _dot(f0["vE"], f0["bgb"]), _dot(f0["vE"], f0["vgb"])
    D = 1.0 - 0.5 * dt * a
    G0 = _gamma(f0, up, mu)
    upr = up * (1.0 + 0.5 * dt * a) + qm * dt * f0["Epar"] + 0.5 * dt * G0 * gg
    if opt == "mirror":
        upr = upr - dt * mu * _dot(f0["b"], f0["gB"]) / (G0 * f0["kap"])
    k1 = 0.25 * dt * dt * gg * gg - D * D / f0["kap"] ** 2
    k2 = upr * dt * gg
    k3 = upr * upr + (1.0 + 2.0 * mu * f0["Bm"] * f0["kap"]) * D * D
    disc = k2 * k2 - 4.0 * k1 * k3
    sg = torch.where(k2 >= 0, 1.0, -1.0)
    q = -0.5 * (k2 + sg * torch.sqrt(disc))
    G1 = torch.where(q != 0, torch.maximum(q / k1, k3 / q), q / k1)
    ok = (k1 < 0) & (disc >= 0) & (G1 >= 1)
    upn = (upr + 0.5 * dt * G1 * gg) / D
    Vn = _vel(f0, qm, upn, mu, opt)
    V, d = Vn, torch.zeros_like(x)
    live = torch.ones_like(ok)
    for k in range(iters or 16):
        nd_ = 0.5 * dt * (Vn + V)[:nd]
        if iters:
            d = nd_
        else:
            done = ((nd_ - d).abs().amax(0) < 1e-7)
            d = torch.where(live, nd_, d)
            live = live & ~done
            if not bool(live.any()):
                break
        if k + 1 < (iters or 16):
            Vk = _vel(_frame(_gather(rec, dims, x + d), opt), qm, upn, mu, opt)
            V = Vk if iters else torch.where(live, Vk, V)
    f = _frame(_gather(rec, dims, x + 0.5 * d), opt)
    Gp = _gamma(f, upn, mu)
    if opt == "phase":
        ph = -qm * f["Bm"] * dt / (f["kap"] * Gp)
        bpg = torch.cos(ph) * bpg + torch.sin(ph) * _cross(f["b"], bpg)
    un = upn * f["b"] + (f["vE"] + _vc(f, qm, upn, Gp)) * Gp
    un = un + torch.sqrt(2.0 * mu * f["Bm"] * f["kap"]) * bpg
    ok = ok & torch.isfinite(un).all(0) & torch.isfinite(d).all(0)   # v_E < c all along
    return ok, un, d, 0.5 * (Vn + V)[2]


def _boris(F, u, qm, dt, nd):
    h = 0.5 * qm * dt
    um = u + h * F[0]
    t = h * F[1] / torch.sqrt(1.0 + _dot(um, um))
    un = um + 2.0 / (1.0 + _dot(t, t)) * _cross(um + _cross(um, t), t) + h * F[0]
    v = un / torch.sqrt(1.0 + _dot(un, un))
    return un, dt * v[:nd], v[2]


def _step(rec, dims, x, u, dxp, qm, p, opt):
    """One coupled step: the switch, then either branch."""
    F0 = _gather(rec, dims, x)
    Bm, Em = torch.sqrt(_dot(F0[1], F0[1])), torch.sqrt(_dot(F0[0], F0[0]))
    G = torch.sqrt(1.0 + _dot(u, u))
    gca = (G < p["f_rho"] * p["dl"] * qm.abs() * Bm) & (Em < p["f_E"] * Bm)
    un, d, vz = _boris(F0, u, qm, p["dt"], len(dims))
    ok, ug, dg, vg = _gca(rec, dims, x, u, dxp, qm, p["dt"], F0, opt, 0)
    ok = ok & gca
    un, d, vz = torch.where(ok, ug, un), torch.where(ok, dg, d), torch.where(ok, vg, vz)
    L = torch.tensor([float(v) for v in dims], device=DEV, dtype=F64)[:, None]
    xn = x + d
    xn = torch.where(xn < 0, xn + L, xn)
    return torch.where(xn >= L, xn - L, xn), un, d, vz


def _deposit(J, dims, x, d, Q, vz, dt):
    """Adds the time-averaged current of cloud-in-cell particles moving from x
    by d over the step to J (3, nodes); pieces between cell faces."""
    nd = len(dims)
    s0 = x
    cr = []
    for k in range(nd):       # at most one face per axis (|d| < 1)
        face = torch.where(d[k] > 0, torch.floor(s0[k]) + 1.0, torch.floor(s0[k]))
        t = (face - s0[k]) / d[k]
        cr.append(torch.where((t > 0) & (t < 1) & (d[k] != 0), t, torch.ones_like(t)))
    cuts = torch.sort(torch.stack(cr), 0).values
    ta = torch.zeros_like(vz)
    for i in range(nd + 1):
        tb = cuts[i] if i < nd else torch.ones_like(vz)
        cell = torch.floor(s0 + d * (0.5 * (ta + tb)))
        m, D = s0 + d * (0.5 * (ta + tb)) - cell, d * (tb - ta)
        idx = [[torch.remainder(cell[k].long() + o, dims[k]) for o in (0, 1)] for k in range(nd)]

        def add(c, offs, val):
            lin = 0
            for k in reversed(range(nd)):
                lin = lin * dims[k] + idx[k][offs[k]]
            J[c].index_add_(0, lin, val)

        for c in range(nd):
            others = [k for k in range(nd) if k != c]
            cr2 = D[others[0]] * D[others[1]] / 12.0 if nd == 3 else 0.0
            for o in range(1 << (nd - 1)):
                w, offs, sgn = 1.0, [0] * nd, 1.0
                for j, k in enumerate(others):
                    hi = (o >> j) & 1
                    offs[k] = hi
                    w = w * (m[k] if hi else 1.0 - m[k])
                    sgn = sgn * (1.0 if hi else -1.0)
                add(c, offs, Q * D[c] / dt * (w + sgn * cr2))
        if nd == 2:
            for o in range(4):
                hi = [o & 1, o >> 1]
                w = (m[0] if hi[0] else 1.0 - m[0]) * (m[1] if hi[1] else 1.0 - m[1])
                sgn = 1.0 if hi[0] == hi[1] else -1.0
                add(2, hi, Q * vz * (tb - ta) * (w + sgn * D[0] * D[1] / 12.0))
        ta = tb


def _records(f):
    comps = list(f["E"]) + list(f["B"]) + (list(f["dB"]) if f["dB"] is not None else [])
    return torch.stack([t.reshape(-1) for t in comps], 1).contiguous()


def _exact_flat(c, seed):
    f, st, p = _flat_inputs(c, seed)
    rec = _records(f)
    dims = (c["nx"], c["ny"]) if c["nz"] == 1 else (c["nx"], c["ny"], c["nz"])
    J = torch.zeros((3, rec.shape[0]), device=DEV, dtype=F64) if c["kind"] == "pic" else None
    qms = torch.tensor(p["qm"], device=DEV, dtype=F64)
    out = {k: torch.empty_like(st[k]) for k in ("x", "u", "dxp")}
    for a in range(0, c["n"], CHUNK):
        sl = slice(a, min(c["n"], a + CHUNK))
        x, u, d = st["x"][:, sl], st["u"][:, sl], st["dxp"][:, sl]
        spc = (st["flags"][sl] >> gcb.SPECIES_SHIFT).long()
        for k in range(c["steps"]):
            x0 = x
            x, u, d, vz = _step(rec, dims, x, u, d, qms[spc], p, c["option"])
            if J is not None and k == c["steps"] - 1:
                Q = torch.tensor([-1.0, 1.0], device=DEV, dtype=F64)[spc]
                _deposit(J, dims, x0, d, Q, vz, p["dt"])
        out["x"][:, sl], out["u"][:, sl], out["dxp"][:, sl] = x, u, d
    out["flags"] = None
    if J is not None:
        out["J"] = J.reshape((3,) + tuple(reversed(dims)))
    return out


def _exact_adjoint(c, seed):
    f, st, p = _flat_inputs(c, seed)
    base, pat, amps = _mode_records(c, seed)
    dims = (c["nx"], c["ny"])
    L = torch.tensor([float(v) for v in dims], device=DEV, dtype=F64)[:, None]
    leaf = [t.clone().requires_grad_() for t in (st["x"], st["u"], st["dxp"])]
    rec = (base.double() + amps @ pat.double()).reshape(-1, 12).requires_grad_()
    qms = torch.tensor(p["qm"], device=DEV, dtype=F64)
    qm = qms[(st["flags"] >> gcb.SPECIES_SHIFT).long()]
    x, u, d = leaf
    for _ in range(c["steps"]):      # strongly magnetized throughout: guiding-center steps
        F0 = _gather(rec, dims, x)
        _, u, d, _ = _gca(rec, dims, x, u, d, qm, p["dt"], F0, "plain", c["iters"])
        x = x + d
        x = x - L * torch.floor(x.detach() / L)
    loss = (torch.sqrt(1.0 + (u * u).sum(0)) - 1.0).sum() + x.sum()
    gx, gu, gd, gr = torch.autograd.grad(loss, leaf + [rec])
    return dict(x=x.detach(), u=u.detach(), dxp=d.detach(), gx=gx, gu=gu, gdxp=gd,
                gamps=pat.double() @ gr.reshape(-1))


# ---- Kerr-Schild
def _metric(a, r, th, derivs=True):
    s, co = torch.sin(th), torch.cos(th)
    s2, a2 = s * s, a * a
    rho2 = r * r + a2 * co * co
    z = 2.0 * r / rho2
    P = r * r + a2 + z * a2 * s2
    m = dict(alpha=1.0 / torch.sqrt(1.0 + z), br=z / (1.0 + z), grr=P / ((1.0 + z) * rho2),
             grp=a / rho2, gtt=1.0 / rho2, gpp=1.0 / (rho2 * s2), drr=1.0 + z,
             drp=-a * (1.0 + z) * s2, dtt=rho2, dpp=P * s2,
             sg=rho2 * s * torch.sqrt(1.0 + z))
    if derivs:
        dm = {k: [] for k in ("alpha", "br", "grr", "grp", "gtt", "gpp")}
        for i in range(2):
            drho = 2.0 * r if i == 0 else -2.0 * a2 * s * co
            dz = (2.0 / rho2 if i == 0 else 0.0) - 2.0 * r * drho / rho2 ** 2
            ds2 = 0.0 if i == 0 else 2.0 * s * co
            dP = (2.0 * r if i == 0 else 0.0) + a2 * (dz * s2 + z * ds2)
            dm["alpha"].append(-0.5 * dz * (1.0 + z) ** -1.5)
            dm["br"].append(dz / (1.0 + z) ** 2)
            dm["grr"].append(m["grr"] * (dP / P - dz / (1.0 + z) - drho / rho2))
            dm["grp"].append(-a * drho / rho2 ** 2)
            dm["gtt"].append(-drho / rho2 ** 2)
            dm["gpp"].append(-m["gpp"] * (drho / rho2 + ds2 / s2))
        m["d"] = dm
    return m


def _raise(m, u):
    return torch.stack([m["grr"] * u[0] + m["grp"] * u[2], m["gtt"] * u[1],
                        m["grp"] * u[0] + m["gpp"] * u[2]])


def _lower(m, v):
    return torch.stack([m["drr"] * v[0] + m["drp"] * v[2], m["dtt"] * v[1],
                        m["drp"] * v[0] + m["dpp"] * v[2]])


def _kgather(K, x):
    s = (torch.log(x[0]) - K["logr0"]) / K["dlogr"]
    q = x[1] / K["dth"]
    i = torch.floor(s).clamp(0, K["nr"] - 2)
    j = torch.floor(q).clamp(0, K["nth"] - 2)
    tr, tt = s - i, q - j
    i, j = i.long(), j.long()
    out = 0.0
    for o in range(4):
        w = (tr if o & 1 else 1.0 - tr) * (tt if o >> 1 else 1.0 - tt)
        out = out + w * K["rec"].index_select(0, (j + (o >> 1)) * K["nr"] + i + (o & 1)).t()
    return out[:3], out[3:6], j * (K["nr"] - 1) + i


def _kframe(K, x, derivs):
    m = _metric(K["a"], x[0], x[1], derivs)
    D, B, cell = _kgather(K, x)
    Bd = _lower(m, B)
    B2 = _dot(Bd, B)
    Bm = torch.sqrt(B2)
    vE = m["sg"] * _cross(D, B) / B2
    v2 = _dot(vE, _raise(m, vE))
    return dict(m=m, D=D, B=B, Bm=Bm, bdn=Bd / Bm, bup=B / Bm, vE=vE, ok=v2 < 1.0,
                kap=1.0 / torch.sqrt(torch.where(v2 < 1.0, 1.0 - v2, torch.ones_like(v2))),
                Dpar=_dot(D, Bd / Bm), cell=cell)


def _force(m, u, G):
    d, g = m["d"], []
    for i in range(2):
        uu = (d["grr"][i] * u[0] ** 2 + 2.0 * d["grp"][i] * u[0] * u[2] + d["gtt"][i] * u[1] ** 2
              + d["gpp"][i] * u[2] ** 2)
        g.append(-G * d["alpha"][i] + u[0] * d["br"][i] - 0.5 * m["alpha"] / G * uu)
    return torch.stack(g + [torch.zeros_like(G)])


def _velocity(m, w):
    v = m["alpha"] * _raise(m, w)
    return torch.stack([v[0] - m["br"], v[1], v[2]])


def _kick(K, x, u, qm, dt):
    """Boris kick over alpha dt / 2 in the global basis (the local-frame kick
    is the same map)."""
    m = _metric(K["a"], x[0], x[1], False)
    D, B, _ = _kgather(K, x)
    h = 0.25 * qm * dt * m["alpha"]
    Dd = _lower(m, D)
    um = u + h * Dd
    v = _raise(m, um)
    t = h * B / torch.sqrt(1.0 + _dot(um, v))
    w = um + m["sg"] * _cross(v, t)
    un = um + 2.0 / (1.0 + _dot(t, _lower(m, t))) * m["sg"] * _cross(_raise(m, w), t)
    return un + h * Dd


def _kerr_step(K, x, u, qm, p):
    dt, tol = p["dt"], p["gca_tol"]
    f0 = _kframe(K, x, False)
    m0 = f0["m"]
    G = torch.sqrt(1.0 + _dot(u, _raise(m0, u)))
    Em = torch.sqrt(_dot(_lower(m0, f0["D"]), f0["D"]))
    gca = f0["ok"] & (G < p["f_rho"] * K["dl"][f0["cell"]] * abs(qm) * f0["Bm"]) & (Em < f0["Bm"])
    # guiding-center branch
    up = _dot(u, f0["bup"])
    ug = u - up * f0["bdn"] - f0["vE"] * G
    uperp = torch.sqrt(_dot(ug, _raise(m0, ug)))
    bpg, mu = ug / uperp, uperp ** 2 / (2.0 * f0["Bm"] * f0["kap"])
    u1 = up + 0.5 * dt * m0["alpha"] * qm * f0["Dpar"]
    R, w, live, ok = x, u1, torch.ones_like(gca), f0["ok"]
    for _ in range(16):
        f = _kframe(K, 0.5 * (R + x), True)
        ok = ok & (f["ok"] | ~live)
        ub, P = 0.5 * (w + u1), 2.0 * mu * f["Bm"] * f["kap"]
        Gm = f["kap"] * torch.sqrt(1.0 + ub * ub + P)
        V = _velocity(f["m"], ub / Gm * f["bdn"] + f["vE"])
        uf = ub * f["bdn"] + f["vE"] * Gm + torch.sqrt(P) * bpg
        Rn, wn = x + dt * V, u1 + dt * _dot(_force(f["m"], uf, Gm), f["bup"])
        res = torch.maximum((Rn - R).abs().amax(0), (wn - w).abs())
        R, w = torch.where(live, Rn, R), torch.where(live, wn, w)
        live = live & ~(res < tol)
        if not bool(live.any()):
            break
    f1 = _kframe(K, R, False)
    up = w + 0.5 * dt * f1["m"]["alpha"] * qm * f1["Dpar"]
    P = 2.0 * mu * f1["Bm"] * f1["kap"]
    ugc = up * f1["bdn"] + f1["vE"] * (f1["kap"] * torch.sqrt(1.0 + up * up + P))
    ugc = ugc + torch.sqrt(P) * bpg
    take = gca & ok & f1["ok"]
    # full-motion branch
    u1 = _kick(K, x, u, qm, dt)
    y, w, live = x, u1, torch.ones_like(gca)
    for _ in range(16):
        xb, ub = 0.5 * (y + x), 0.5 * (w + u1)
        m = _metric(K["a"], xb[0], xb[1])
        Gm = torch.sqrt(1.0 + _dot(ub, _raise(m, ub)))
        yn, wn = x + dt * _velocity(m, ub / Gm), u1 + dt * _force(m, ub, Gm)
        res = torch.maximum((yn - y).abs().amax(0), (wn - w).abs().amax(0))
        y, w = torch.where(live, yn, y), torch.where(live, wn, w)
        live = live & ~(res < tol)
        if not bool(live.any()):
            break
    w = _kick(K, y, w, qm, dt)
    return torch.where(take, R, y), torch.where(take, ugc, w)


def _exact_kerr(c, seed):
    f, p, x, u = _kerr_inputs(c, seed)
    comps = [torch.as_tensor(t, device=DEV, dtype=F64).reshape(-1)
             for t in list(f["D"]) + list(f["B"])]
    nr, nth, a = c["nx"], c["ny"], float(f["a"])
    K = dict(a=a, rec=torch.stack(comps, 1).contiguous(), nr=nr, nth=nth,
             logr0=float(f["logr0"]), dlogr=float(f["dlogr"]), dth=math.pi / (nth - 1))
    # cell sizes: square root of the area, 4 x 4 Gauss points
    gx, gw = [0.3399810435848563, 0.8611363115940526], [0.6521451548625461, 0.3478548451374538]
    r = torch.exp(K["logr0"] + K["dlogr"] * torch.arange(nr, device=DEV, dtype=F64))
    t = K["dth"] * torch.arange(nth, device=DEV, dtype=F64)
    area = 0.0
    for X, W in zip([-gx[1], -gx[0], gx[0], gx[1]], [gw[1], gw[0], gw[0], gw[1]]):
        for Y, V in zip([-gx[1], -gx[0], gx[0], gx[1]], [gw[1], gw[0], gw[0], gw[1]]):
            rr = (0.5 * (r[:-1] + r[1:]) + 0.5 * X * (r[1:] - r[:-1]))[None, :]
            tt = (0.5 * (t[:-1] + t[1:]) + 0.5 * Y * (t[1:] - t[:-1]))[:, None]
            rho2 = rr * rr + a * a * torch.cos(tt) ** 2
            area = area + W * V * torch.sqrt((1.0 + 2.0 * rr / rho2) * rho2)
    area = area * 0.25 * (r[1:] - r[:-1])[None, :] * (t[1:] - t[:-1])[:, None]
    K["dl"] = torch.sqrt(area).reshape(-1)
    qm = float(p["qm"][0])
    frozen = torch.zeros(c["n"], device=DEV, dtype=torch.bool)
    for _ in range(c["steps"]):
        xs, us = [], []
        for i in range(0, c["n"], CHUNK):
            y, w = _kerr_step(K, x[:, i:i + CHUNK], u[:, i:i + CHUNK], qm, p)
            xs.append(y)
            us.append(w)
        y, w = torch.cat(xs, 1), torch.cat(us, 1)
        for bad, ref in ((y[1] < 0, -y[1]), (y[1] > math.pi, 2 * math.pi - y[1])):
            y = torch.stack([y[0], torch.where(bad, ref, y[1]),
                             torch.where(bad, y[2] + math.pi, y[2])])
            w = torch.stack([w[0], torch.where(bad, -w[1], w[1]), w[2]])
        y = torch.stack([y[0], y[1], torch.remainder(y[2], 2 * math.pi)])
        x, u = torch.where(frozen, x, y), torch.where(frozen, u, w)
        frozen = frozen | (x[0] < float(p["r_in"])) | (x[0] > float(p["r_out"]))
    return dict(x=x, u=u, flags=None)


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    if case["kind"] == "kerr":
        return _exact_kerr(case, seed)
    return _exact_flat(case, seed)
