"""Work that users of this library have it do, as cases that can be timed.

Fields are random-phase solenoidal k^-5/3 fields with unit rms per component on the
periodic box [0, 2 pi)^3, particles are uniform in the box with FP64 positions, the
coefficients and results are those of the public Python API.  `exact` restates the
method in 64 bits with torch alone: the periodic (1/6, 4/6, 1/6) solves in Fourier
space, the 64-term sums, their derivatives and adjoint, and Heun's method.

A tracked particle set is stored in bin order and its order inside a bin is left open
by the library, so the tracking cases return positions and velocities by particle
label, as a program does that writes trajectories.
"""
import math

import torch

import paper_2005_13193_gb300 as ps

TWO_PI = 2.0 * math.pi
BRICK = (8, 8, 8)
STORE = {"f32": torch.float32, "f64": torch.float64, "f32x4": ps.F32X4, "bf16x4": ps.BF16X4,
         "f16x4": ps.F16X4}


def listed():
    return [
        # the smallest use: a field comes in, its coefficients, one interpolation and one
        # binned Heun step of a few thousand particles; launches and latency count
        dict(name="tiny_32", kind="tiny", nx=32, ny=32, nz=32, np=4096, dt=1e-3),
        # a simulation's step hands over a new velocity field: coefficients as nodes, the
        # storage that tracking uses
        dict(name="solve_512_nodes", kind="solve", nx=512, ny=512, nz=512, ncomp=3, store="f32x4"),
        # a box whose sides are no powers of two, planar coefficients (the default storage)
        dict(name="solve_ragged", kind="solve", nx=250, ny=200, nz=150, ncomp=3, store="f32"),
        # rows over 512 values, the large workload's sequence (a new field, its coefficients,
        # one binned Heun step at 0.083 particles per cell) at an eighth of its size
        dict(name="scale_768", kind="scale", nx=768, ny=768, nz=768, np=37_500_000,
             store="f32x4", dt=1e-3),
        # the same sequence with 16-bit coefficients, an ordinary size
        dict(name="scale_256_f16", kind="scale", nx=256, ny=256, nz=256, np=1_400_000,
             store="f16x4", dt=1e-3),
        # velocities at 16.8 M particles kept in bin order
        dict(name="interp_512", kind="interp", nx=512, ny=512, nz=512, np=1 << 24,
             store="f32x4"),
        # a one-off look-up at particles in no order, default storage, no bins
        dict(name="scattered_128", kind="scattered", nx=128, ny=128, nz=128, np=250_000,
             ncomp=3, store="f32"),
        # Lagrangian statistics: bins, velocity gradients, second derivatives and the
        # acceleration from two fields at the same particles
        dict(name="derivatives_256", kind="derivatives", nx=256, ny=256, nz=256, np=4_000_000,
             store="f32x4", dt=1e-2),
        # the production loop: re-binned Heun steps through a frozen field
        dict(name="track_512", kind="track", nx=512, ny=512, nz=512, np=1 << 24, store="f32x4",
             unsteady=False, steps=4, dt=1e-3),
        # tracking between two snapshots of a field, default storage, a ragged box
        dict(name="track_unsteady", kind="track", nx=180, ny=150, nz=132, np=500_000,
             store="f32", unsteady=True, steps=2, dt=2e-3),
        # differentiable interpolation: forward, and the gradients for positions and field
        dict(name="autograd_256", kind="autograd", nx=256, ny=256, nz=256, np=4_000_000),
        # many independent fields with particle sets of uneven sizes, solved and advanced
        # together from one captured graph
        dict(name="batch_16", kind="batch", fields=16, mix=3000, steps=4, store="f32", dt=1e-3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """Three extents: a cube of a common size, or ragged ones."""
    if rng.random() < 0.4:
        common = [e for e in (32, 64, 96, 128, 192, 256, 320, 384, 512, 640, 768) if lo <= e <= hi]
        e = rng.choice(common)
        return dict(nx=e, ny=e, nz=e)
    return dict(nx=_log(rng, lo, hi), ny=_log(rng, lo, hi), nz=_log(rng, lo, hi))


def draw(rng):
    kind = rng.choice(["tiny", "solve", "scale", "interp", "scattered", "derivatives", "track",
                       "autograd", "batch"])
    if kind == "tiny":
        return dict(kind=kind, np=_log(rng, 500, 20_000), dt=1e-3, **_box(rng, 16, 64))
    if kind == "solve":
        store = rng.choice(["f32", "f32x4"])
        ncomp = 3 if store == "f32x4" else rng.choice([1, 3])
        return dict(kind=kind, store=store, ncomp=ncomp, **_box(rng, 48, 512))
    if kind == "scale":
        c = dict(kind=kind, store=rng.choice(["f32x4", "bf16x4", "f16x4"]), dt=1e-3,
                 **_box(rng, 96, 640))
        cells = c["nx"] * c["ny"] * c["nz"]
        return c | dict(np=max(10_000, int(cells * rng.uniform(0.04, 0.12))))
    if kind == "interp":
        return dict(kind=kind, np=_log(rng, 50_000, 1 << 24),
                    store=rng.choice(["f32x4", "f32", "bf16x4"]), **_box(rng, 64, 384))
    if kind == "scattered":
        return dict(kind=kind, np=_log(rng, 10_000, 4_000_000), ncomp=rng.choice([1, 3]),
                    store=rng.choice(["f32", "f64"]), **_box(rng, 48, 256))
    if kind == "derivatives":
        return dict(kind=kind, np=_log(rng, 50_000, 4_000_000), dt=1e-2,
                    store=rng.choice(["f32x4", "f32", "f16x4"]), **_box(rng, 64, 256))
    if kind == "track":
        return dict(kind=kind, np=_log(rng, 20_000, 8_000_000),
                    store=rng.choice(["f32x4", "f32", "bf16x4"]), unsteady=rng.random() < 0.4,
                    steps=rng.choice([1, 2, 4]), dt=rng.choice([1e-3, 2e-3]),
                    **_box(rng, 64, 384))
    if kind == "autograd":
        return dict(kind=kind, np=_log(rng, 5_000, 4_000_000), **_box(rng, 48, 256))
    return dict(kind="batch", fields=rng.choice([3, 6, 12, 16]), mix=rng.randrange(1, 10_000),
                steps=rng.choice([2, 4]), store=rng.choice(["f32", "f32x4"]), dt=1e-3)


# ------------------------------------------------------------------ inputs --

def _n(c):
    return (c["nx"], c["ny"], c["nz"])


def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + k)


def _field(n, ncomp, gen, dtype=torch.float32):
    """[ncomp][nz][ny][nx]: white noise shaped to k^-5/3 for 1 <= |k| <= min(n) / 3,
    made solenoidal when it has three components, unit rms."""
    nx, ny, nz = n
    rf = torch.float64 if dtype == torch.float64 else torch.float32
    kx = torch.arange(nx // 2 + 1, device="cuda", dtype=rf)
    ky = torch.fft.fftfreq(ny, d=1.0 / ny, device="cuda", dtype=rf).view(ny, 1)
    kz = torch.fft.fftfreq(nz, d=1.0 / nz, device="cuda", dtype=rf).view(nz, 1, 1)
    k2 = kx * kx + ky * ky + kz * kz
    kmax = min(n) // 3
    amp = torch.where((k2 >= 1) & (k2 <= kmax * kmax), k2.clamp(min=1).pow(-11.0 / 12.0), 0.0)
    spec = [torch.fft.rfftn(torch.randn((nz, ny, nx), generator=gen, device="cuda", dtype=rf))
            * amp for _ in range(ncomp)]
    del amp
    if ncomp == 3:
        div = (kx * spec[0] + ky * spec[1] + kz * spec[2]) / k2.clamp(min=1)
        for k, s in zip((kx, ky, kz), spec):
            s -= k * div
        del div
    out = torch.empty((ncomp, nz, ny, nx), device="cuda", dtype=dtype)
    for i in range(ncomp):
        f = torch.fft.irfftn(spec[i], s=(nz, ny, nx))
        spec[i] = None
        out[i] = f / torch.linalg.vector_norm(f) * math.sqrt(f.numel())
    return out


def _particles(count, gen):
    return torch.rand((3, count), generator=gen, device="cuda", dtype=torch.float64) * TWO_PI


def _in_bin_order(n, pos):
    """The positions sorted by brick (stable, so the same from run to run)."""
    key = torch.zeros(pos.shape[1], device="cuda", dtype=torch.int64)
    for d in (2, 1, 0):
        nb = -(-n[d] // BRICK[d])
        cell = torch.floor(pos[d] * (n[d] / TWO_PI)).long() % n[d]
        key = key * nb + cell // BRICK[d]
    return pos[:, torch.sort(key, stable=True).indices].contiguous()


def _inputs(c, seed):
    """The field(s) and particles of a case, from the seed alone."""
    g = _gen(seed, 0)
    kind = c["kind"]
    if kind == "batch":
        edges, nps = _mix(c)
        return dict(fields=[_field((e, e, e), 3, g) for e in edges],
                    pos=torch.cat([_particles(m, g) for m in nps], dim=1))
    n = _n(c)
    i = dict(field=_field(n, c.get("ncomp", 3), g,
                          torch.float64 if kind == "tiny" or c.get("store") == "f64"
                          else torch.float32))
    if kind == "derivatives" or c.get("unsteady"):
        i["later"] = 0.98 * i["field"] + 0.2 * _field(n, 3, g)
    if kind != "solve":
        i["pos"] = _particles(c["np"], _gen(seed, 1))
        if kind in ("interp", "track", "tiny", "scale"):
            i["pos"] = _in_bin_order(n, i["pos"])
    if kind == "autograd":
        i["g_vel"] = torch.randn((3, c["np"]), generator=_gen(seed, 2), device="cuda")
    return i


def _mix(c):
    """Grid edges and particle counts of a batch: edges uniform over the common sizes,
    counts log-uniform between 10,000 and 2,000,000."""
    g = torch.Generator().manual_seed(c["mix"])
    sizes = (64, 96, 128, 192, 256)
    edges = [sizes[int(k)] for k in torch.randint(0, 5, (c["fields"],), generator=g)]
    u = torch.rand(c["fields"], generator=g, dtype=torch.float64)
    nps = [int(round(math.exp(math.log(1e4) + float(v) * math.log(200.0)))) for v in u]
    return edges, nps


def prepare(case, seed):
    c = case
    i = _inputs(c, seed)
    kind = c["kind"]
    s = dict(case=c, **i)
    if kind == "batch":
        edges, nps = _mix(c)
        s["plan"] = ps.BatchPlan([(e, e, e) for e in edges], nps, coef_dtype=STORE[c["store"]],
                                 brick=BRICK)
        s["plan"].workspace()
        s["sf"] = [ps.SplineField.from_field(f, STORE[c["store"]]) for f in i["fields"]]
        s["ids"] = torch.arange(s["pos"].shape[1], device="cuda", dtype=torch.int64)
        s["vel"] = torch.empty((3, s["pos"].shape[1]), device="cuda")
        return s
    n = _n(c)
    if kind == "autograd":
        s["pos"].requires_grad_()
        s["field"].requires_grad_()
        return s
    store = STORE[c.get("store", "f32")]
    s["sf"] = ps.SplineField.from_field(i["field"], store)
    need = ps.ps_spline_coeffs_workspace_size(n, s["sf"].ncomp, store)
    if kind in ("tiny", "solve", "scale"):
        s["ws"] = ps.workspace(need) if need else None
    else:
        del s["field"]
    if "later" in i:
        s["later"] = ps.SplineField.from_field(i["later"], store)
    if kind == "interp":
        s["bins"] = ps.bin_particles(n, BRICK, s["pos"], want_perm=False)
    if kind in ("tiny", "scale", "track"):
        s["tracker"] = ps.Tracker(s["sf"], s["pos"], brick=BRICK)
    return s


# --------------------------------------------------------------------- run --

def _by_label(ids, *arrays):
    return [torch.empty_like(a).index_copy_(1, ids, a) for a in arrays]


def run(state):
    s = state
    c = s["case"]
    kind = c["kind"]
    if kind == "solve":
        return ps.SplineField.from_field(s["field"], out=s["sf"], ws=s["ws"]).coef
    if kind == "interp":
        return s["sf"].interp(s["pos"], bins=s["bins"])
    if kind == "scattered":
        return s["sf"].interp(s["pos"])
    if kind == "derivatives":
        bins = ps.bin_particles(_n(c), BRICK, s["pos"])
        vel, grad = s["sf"].interp(s["pos"], grad=True, bins=bins)
        hess = s["sf"].hessian(s["pos"], bins=bins)
        acc = s["sf"].acceleration(s["pos"], later=s["later"], dt_field=c["dt"], bins=bins)
        return dict(vel=vel, grad=grad, hess=hess, acc=acc, offsets=bins.offsets,
                    bin_of=bins.bin_of)
    if kind == "autograd":
        vel = ps.interp_autograd(s["pos"], s["field"])
        g_pos, g_field = torch.autograd.grad(vel, (s["pos"], s["field"]), s["g_vel"])
        return dict(vel=vel, g_pos=g_pos, g_field=g_field)
    if kind == "batch":
        s["plan"].run(list(zip(s["fields"], s["sf"])), s["pos"], c["steps"], c["dt"],
                      ids=s["ids"], vel=s["vel"])
        return _by_label(s["ids"], s["pos"], s["vel"])
    tr = s["tracker"]
    if kind == "track":
        for _ in range(c["steps"]):
            tr.step(c["dt"], field_np1=s.get("later"))
        return _by_label(tr.ids, tr.pos, tr.vel)
    # tiny, scale: a new field, its coefficients, then the particles
    ps.SplineField.from_field(s["field"], out=s["sf"], ws=s["ws"])
    first = [s["sf"].interp(tr.pos)] if kind == "tiny" else []
    if first:
        first = _by_label(tr.ids, *first)
    tr.step(c["dt"])
    return first + _by_label(tr.ids, tr.pos, tr.vel)


# -------------------------------------------------------------------- work --

def _coef_bytes(n, ncomp, store):
    """Coefficients at their planar size (three components also where nodes hold a
    fourth, zero one)."""
    size = {"f32": 4, "f64": 8, "f32x4": 4, "bf16x4": 2, "f16x4": 2}[store]
    return ncomp * size * (n[0] + 3) * (n[1] + 3) * (n[2] + 3)


def work(case):
    c = case
    kind = c["kind"]
    if kind == "batch":
        edges, nps = _mix(c)
        b = f = 0
        for e, m in zip(edges, nps):
            k = _coef_bytes((e, e, e), 3, "f32")
            b += 12 * e ** 3 + k + c["steps"] * k + m * 60 * c["steps"] + m * 24
            f += 3 * e ** 3 * 15 + m * c["steps"] * 2 * 600
        return dict(bytes=b, flops=f)
    n = _n(c)
    cells = n[0] * n[1] * n[2]
    ncomp = c.get("ncomp", 3)
    coef = _coef_bytes(n, ncomp, c.get("store", "f32"))
    m = c.get("np", 0)
    # two first-order recursions and a gain per value and axis; a stencil sum is
    # 84 multiply-adds per component, and each particle needs 3 x 4 weights
    solve = (cells * ncomp * (8 if kind == "tiny" or c.get("store") == "f64" else 4) + coef,
             15 * ncomp * cells)
    sums = 168 * ncomp + 60
    if kind == "solve":
        return dict(bytes=solve[0], flops=solve[1])
    touched = min(coef, m * 64 * coef // cells)  # a sparse set reads less than all
    if kind in ("interp", "scattered"):
        return dict(bytes=touched + m * (24 + 4 * ncomp), flops=m * sums)
    if kind == "derivatives":
        # bins; values and gradients; second derivatives; two fields' values
        return dict(bytes=m * (24 + 4) + 2 * touched + m * (24 + 12 + 36 + 72 + 12),
                    flops=m * (12 * sums))
    if kind == "autograd":
        # forward; both gradients: positions, cotangent in, position gradients out,
        # the field gradient's scatter and its solve
        return dict(bytes=solve[0] + touched + m * 36 + touched + m * (24 + 12 + 24)
                    + 12 * cells * 2, flops=2 * solve[1] + m * 6 * sums)
    step = touched + m * (24 + 24 + 12)
    if c.get("unsteady"):
        step += touched
    if kind == "track":
        return dict(bytes=c["steps"] * step + m * 36, flops=c["steps"] * m * 2 * sums)
    extra = touched + m * 36 if kind == "tiny" else 0
    return dict(bytes=solve[0] + extra + step + m * 36, flops=solve[1] + m * 3 * sums)


# ------------------------------------------------------------------- exact --

def _coef64(field):
    """Spline coefficients in 64 bits: the periodic (1/6, 4/6, 1/6) systems divided out
    in Fourier space.  [ncomp][nz][ny][nx]."""
    out = torch.empty(field.shape, device="cuda", dtype=torch.float64)
    nz, ny, nx = field.shape[1:]

    def eig(n, k):
        return (4 + 2 * torch.cos(TWO_PI * k / n)) / 6

    ex = eig(nx, torch.arange(nx // 2 + 1, device="cuda", dtype=torch.float64))
    ey = eig(ny, torch.arange(ny, device="cuda", dtype=torch.float64)).view(ny, 1)
    ez = eig(nz, torch.arange(nz, device="cuda", dtype=torch.float64)).view(nz, 1, 1)
    for i in range(field.shape[0]):
        s = torch.fft.rfftn(field[i].double())
        s /= ex
        s /= ey
        s /= ez
        out[i] = torch.fft.irfftn(s, s=(nz, ny, nx))
        del s
    return out


def _weights(t, order):
    if order == 0:
        s = 1 - t
        return [s ** 3 / 6, (3 * t ** 3 - 6 * t ** 2 + 4) / 6,
                (-3 * t ** 3 + 3 * t ** 2 + 3 * t + 1) / 6, t ** 3 / 6]
    if order == 1:
        return [-(1 - t) ** 2 / 2, (3 * t ** 2 - 4 * t) / 2, (-3 * t ** 2 + 2 * t + 1) / 2,
                t ** 2 / 2]
    return [1 - t, 3 * t - 2, 1 - 3 * t, t]


_VALUE = ((0, 0, 0),)
_GRAD = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
_HESS = ((2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1))


def _stencil(n, pos, orders):
    """Node indices per axis and offset, and the weights per axis, order and offset."""
    idx, w = [], []
    for d in range(3):
        s = pos[d] * (n[d] / TWO_PI)
        a = torch.floor(s)
        t = s - a
        idx.append([(a.long() + k - 1) % n[d] for k in range(4)])
        w.append({o: _weights(t, o) for o in {q[d] for q in orders}})
    return idx, w


def _eval64(coef, pos, orders=_VALUE, part=1 << 21):
    """out[order][comp][np]: the 64-term sum with derivative orders (x, y, z)."""
    nz, ny, nx = coef.shape[1:]
    n = (nx, ny, nz)
    flat = coef.reshape(coef.shape[0], -1)
    out = torch.zeros((len(orders), coef.shape[0], pos.shape[1]), device="cuda",
                      dtype=torch.float64)
    for p0 in range(0, pos.shape[1], part):
        x = pos[:, p0:p0 + part]
        idx, w = _stencil(n, x, orders)
        for k in range(4):
            for j in range(4):
                row = (idx[2][k] * ny + idx[1][j]) * nx
                wyz = [w[1][o[1]][j] * w[2][o[2]][k] for o in orders]
                for i in range(4):
                    at = row + idx[0][i]
                    for cc in range(coef.shape[0]):
                        v = flat[cc][at]
                        for q, o in enumerate(orders):
                            out[q, cc, p0:p0 + part] += wyz[q] * w[0][o[0]][i] * v
    for q, o in enumerate(orders):
        out[q] *= math.prod((n[d] / TWO_PI) ** o[d] for d in range(3))
    return out


def _heun64(c0, c1, pos, dt):
    u1 = _eval64(c0, pos)[0]
    u2 = _eval64(c1, pos + dt * u1)[0]
    return pos + 0.5 * dt * (u1 + u2), u1


def _padded64(coef, store):
    """The storage layout: padded index P holds node (P - 1) mod n, rows up to the pitch."""
    ncomp, nz, ny, nx = coef.shape
    n = (nx, ny, nz)
    at = [(torch.arange(n[d] + 3, device="cuda") - 1) % n[d] for d in range(3)]
    rx = ps.coef_row_pitch(nx, STORE[store])
    shape = (nz + 3, ny + 3, rx, 4) if store == "f32x4" else (ncomp, nz + 3, ny + 3, rx)
    out = torch.zeros(shape, device="cuda", dtype=torch.float64)
    for i in range(ncomp):
        v = coef[i][at[2]][:, at[1]][:, :, at[0]]
        if store == "f32x4":
            out[:, :, :nx + 3, i] = v
        else:
            out[i, :, :, :nx + 3] = v
    return out


def exact(case, seed):
    c = case
    i = _inputs(c, seed)
    kind = c["kind"]
    if kind == "batch":
        pos, vel, base = [], [], 0
        for f, m in zip(i["fields"], _mix(c)[1]):
            coef, x = _coef64(f), i["pos"][:, base:base + m]
            for _ in range(c["steps"]):
                x, u = _heun64(coef, coef, x, c["dt"])
            pos.append(x)
            vel.append(u)
            base += m
        return [torch.cat(pos, dim=1), torch.cat(vel, dim=1)]
    coef = _coef64(i["field"])
    if kind == "solve":
        return _padded64(coef, c["store"])
    pos = i["pos"]
    if kind in ("interp", "scattered"):
        return _eval64(coef, pos)[0]
    if kind == "derivatives":
        e = _eval64(coef, pos, _VALUE + _GRAD + _HESS)
        u, grad, hess = e[0], e[1:4], e[4:]
        later = _eval64(_coef64(i["later"]), pos)[0]
        acc = (grad * u.unsqueeze(1)).sum(0) + (later - u) / c["dt"]
        return dict(vel=u, grad=grad.transpose(0, 1).contiguous(),
                    hess=hess.transpose(0, 1).contiguous(), acc=acc, offsets=None, bin_of=None)
    if kind == "autograd":
        e = _eval64(coef, pos, _VALUE + _GRAD)
        g = i["g_vel"].double()
        nz, ny, nx = coef.shape[1:]
        g_field = torch.zeros((3, nz * ny * nx), device="cuda", dtype=torch.float64)
        idx, w = _stencil((nx, ny, nz), pos, _VALUE)
        for k in range(4):
            for j in range(4):
                for q in range(4):
                    at = (idx[2][k] * ny + idx[1][j]) * nx + idx[0][q]
                    ww = w[0][0][q] * w[1][0][j] * w[2][0][k]
                    for cc in range(3):
                        g_field[cc].index_add_(0, at, ww * g[cc])
        return dict(vel=e[0], g_pos=(e[1:4] * g).sum(1),
                    g_field=_coef64(g_field.view(3, nz, ny, nx)))
    if kind == "track":
        c1 = _coef64(i["later"]) if c["unsteady"] else coef
        for _ in range(c["steps"]):
            pos, u = _heun64(coef, c1, pos, c["dt"])
        return [pos, u]
    first = [_eval64(coef, pos)[0]] if kind == "tiny" else []
    return first + list(_heun64(coef, coef, pos, c["dt"]))
