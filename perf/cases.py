"""The work that users of the solver have it do, as timed cases.

`listed()` names them; `draw(rng)` gives more of the same ranges.  Every case
runs through the package's public entry points: `lib.Solver`, `lib.Solver3D`
and `lib.BatchSolver` for the lattices (set the initial moments, advance, take
the moments out), `surrogate` for the network's layers and its gradient.

`exact(case, seed)` is the same computation in 64 bits, written here from the
model's equations in plain torch (whole lattices shifted with torch.roll).
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as Fn

from paper_2101_03055_gb300 import inputs as I
from paper_2101_03055_gb300 import lib
from paper_2101_03055_gb300 import surrogate as S

M = 2  # scalars per lattice: the two of every experiment


def listed():
    return [
        # the validation box: a small lattice, where launches and latency count
        dict(name="taylor_green_64", kind="lattice", flow="box", nx=64, ny=64, storage="fp32", steps=100),
        # the chemotaxis plume of the paper's figures (fits in L2)
        dict(name="plume_512x256", kind="lattice", flow="plume", nx=512, ny=256, storage="fp32", steps=256),
        # the double-diffusive cavity with Soret and Dufour terms
        dict(name="cavity_1024", kind="lattice", flow="cavity", nx=1024, ny=1024, storage="fp32", steps=64),
        # the largest single lattice that is run in earnest, FP32 storage
        dict(name="box_4096", kind="lattice", flow="box", nx=4096, ny=4096, storage="fp32", steps=16),
        # 16-bit storage, chosen where capacity counts; odd sizes
        dict(name="plume_bf16_2001x1203", kind="lattice", flow="plume", nx=2001, ny=1203, storage="bf16", steps=32),
        # scalars in a prescribed velocity (no fluid), walls
        dict(name="cellular_2048", kind="lattice", flow="cellular", nx=2048, ny=2048, storage="fp32", steps=32),
        # three dimensions: a periodic box, ragged sizes
        dict(name="box3d_130x112x96", kind="lattice3d", flow="box", nx=130, ny=112, nz=96, steps=400),
        # a parameter sweep: plumes of uneven sizes in one batch, mode left to the library
        dict(name="sweep_64_plumes", kind="batch", flow="plume", count=64, n=0, steps=64),
        # training data of the surrogate: many small cavities, as generate_steady_states runs them
        dict(name="sweep_512_cavities_64", kind="batch", flow="cavity", count=512, n=64, steps=64),
        # the network's first level on a 256 x 256 lattice, forward
        dict(name="conv_fwd_16x256x256_32_32", kind="conv_fwd", N=16, H=256, W=256, cin=32, cout=32),
        # its deepest level, gradients of input, weights and bias
        dict(name="conv_bwd_16x32x32_256_256", kind="conv_bwd", N=16, H=32, W=32, cin=256, cout=256),
        # loss and all gradients of the network on a training batch
        dict(name="unet_gradient_32x64", kind="unet", N=32, n=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "lattice3d", "batch", "conv_fwd", "conv_bwd", "unet"])
    if kind == "lattice":
        flow = rng.choice(["box", "plume", "cavity", "cellular"])
        storage = "fp32" if flow == "cellular" else rng.choice(["fp32", "fp32", "fp16", "bf16"])
        nx, ny = _log(rng, 48, 4096), _log(rng, 48, 2048)
        steps = max(8, min(256, 100_000_000 // (nx * ny)))
        return dict(kind=kind, flow=flow, nx=nx, ny=ny, storage=storage, steps=steps)
    if kind == "lattice3d":
        nx, ny, nz = (_log(rng, 24, 160) for _ in range(3))
        return dict(kind=kind, flow=rng.choice(["box", "cavity"]), nx=nx, ny=ny, nz=nz,
                    steps=max(50, min(400, 500_000_000 // (nx * ny * nz))))
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind=kind, flow="plume", count=rng.randint(4, 64), n=0, steps=rng.randint(20, 64))
        return dict(kind=kind, flow="cavity", count=_log(rng, 32, 512), n=rng.choice([48, 64, 80]),
                    steps=rng.randint(20, 64))
    if kind == "unet":
        return dict(kind=kind, N=rng.choice([8, 16, 24, 32]), n=rng.choice([32, 48, 64]))
    cin, cout = rng.choice([(16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (64, 128), (128, 128), (192, 64),
                            (128, 256), (384, 128), (256, 256)])
    side = _log(rng, 8, 256)
    top = 16 * 256 * 256 * 32 * 32  # the listed layers' work
    n = max(1, min(rng.randint(1, 32), top // (side * side * cin * cout)))
    w = side if rng.random() < 0.7 else max(8, side - rng.randint(1, 7))
    return dict(kind=kind, N=n, H=side, W=w, cin=cin, cout=cout)


# ---- problems -------------------------------------------------------------------------
_D_BOX = ((0.05, 0.01), (0.005, 0.03))


def _flat(shape, v=0.0):
    """A constant field without its memory (the state comes from the device fields)."""
    return np.broadcast_to(np.float64(v), shape)


def _problem(flow, nx, ny, prm=None):
    fields = dict(phi0=_flat((M, ny, nx), 1.0), u0=_flat((2, ny, nx)), p0=_flat((ny, nx)))
    if flow == "box":  # periodic, constant cross-diffusion
        return I.Problem("box", nx, ny, M, np.array(_D_BOX), 0.1, **fields)
    if flow == "cellular":  # Case 1 in a cellular flow between walls
        hot = I.wall_side(M, I.NOSLIP, [I.DIRICHLET] * M, [1.2] * M)
        cold = I.wall_side(M, I.NOSLIP, [I.DIRICHLET] * M, [0.8] * M)
        return I.Problem("cellular", nx, ny, M, np.array(_D_BOX), 0.1, case1=True, west=hot, east=cold,
                         south=I.wall_side(M), north=I.wall_side(M), **fields)
    if flow == "plume":
        prm = prm or {}
        return I.chemotaxis_plume(8, ny, **prm).replace(nx=nx, **fields)
    prm = prm or dict(Ra=1e5, Pr=0.7, Le=2.0, Nc=1.0, Df=0.5, Sr=0.5)
    return I.ddc_cavity(8, **prm).replace(nx=nx, ny=ny, **_cavity_scale(nx, prm),
                                          **dict(fields, phi0=_flat((M, ny, nx), 0.0)))


def _cavity_scale(n, prm):
    pb = I.ddc_cavity(n, ny=1, **prm)  # lattice coefficients of a cavity n nodes across
    return dict(D=pb.D, nu=pb.nu, beta=pb.beta)


def _grid(nx, ny):
    x = (torch.arange(nx, device="cuda", dtype=torch.float32) + 0.5) / nx
    y = (torch.arange(ny, device="cuda", dtype=torch.float32) + 0.5) / ny
    return x[None, :], y[:, None]


def _fields(flow, nx, ny, gen):
    """Initial moments phi_0, phi_1, u_x, u_y, p on the device, FP32."""
    out = torch.zeros((M + 3, ny, nx), device="cuda", dtype=torch.float32)
    x, y = _grid(nx, ny)
    noise = torch.rand((M, ny, nx), generator=gen, device="cuda") * 2 - 1
    pi = math.pi
    if flow == "box":
        u0, v0 = 0.02, 0.02 * ny / nx
        out[:M] = 1 + 0.1 * noise
        out[2] = -u0 * torch.cos(2 * pi * x) * torch.sin(2 * pi * y)
        out[3] = v0 * torch.sin(2 * pi * x) * torch.cos(2 * pi * y)
        out[4] = -0.25 * (u0 ** 2 * torch.cos(4 * pi * x) + v0 ** 2 * torch.cos(4 * pi * y))
        if v0 > 0.05:  # a tall box: start from rest, the discrete velocity set wants small u
            out[2:] = 0
    elif flow == "cellular":
        u0 = 0.05 if ny <= nx else 0.05 * nx / ny
        out[:M] = 1 + 0.1 * noise
        out[2] = u0 * torch.sin(pi * x) * torch.cos(pi * y)
        out[3] = -u0 * (ny / nx) * torch.cos(pi * x) * torch.sin(pi * y)
    elif flow == "plume":
        out[0] = 1 + 0.01 * torch.randn((ny, nx), generator=gen, device="cuda")
        out[1] = 1
    else:  # a developed cavity: conduction profile, noise, a weak circulation
        out[:M] = (1 - x) + 0.05 * noise
        out[2] = 0.01 * torch.sin(pi * x) * torch.cos(pi * y)
        out[3] = -0.01 * torch.cos(pi * x) * torch.sin(pi * y)
    return out


def _fields3(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    r = np.random.default_rng(seed)
    noise = 2 * r.random((M, nz, ny, nx), dtype=np.float32) - 1
    x = ((np.arange(nx) + 0.5) / nx)[None, None, :]
    y = ((np.arange(ny) + 0.5) / ny)[None, :, None]
    z = ((np.arange(nz) + 0.5) / nz)[:, None, None]
    u, p = np.zeros((3, nz, ny, nx)), np.zeros((nz, ny, nx))
    if case["flow"] == "box":
        phi = 1 + 0.1 * noise.astype(np.float64)
        k = 2 * math.pi
        u[0] = 0.02 * np.sin(k * x) * np.cos(k * y) * np.cos(k * z)
        u[1] = -0.02 * np.cos(k * x) * np.sin(k * y) * np.cos(k * z)
    else:
        phi = (1 - x) + 0.05 * noise.astype(np.float64)
    return [np.ascontiguousarray(a.astype(np.float32).astype(np.float64)) for a in (phi, u, p)]


def _problem3(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["flow"] == "box":
        return I.Problem3D("box3d", nx, ny, nz, M, np.array(_D_BOX), 0.1, phi0=_flat((M, nz, ny, nx), 1.0),
                           u0=_flat((3, nz, ny, nx)), p0=_flat((nz, ny, nx)))
    return I.ddc_cavity3d(8).replace(nx=nx, ny=ny, nz=nz, **_cavity_scale(nx, dict(Ra=1e4)),
                                     phi0=_flat((M, nz, ny, nx)), u0=_flat((3, nz, ny, nx)), p0=_flat((nz, ny, nx)))


def _members(case, seed):
    """The instances of a batch: their problems and their fields' sizes."""
    r = np.random.default_rng(seed)
    pbs = []
    for _ in range(case["count"]):
        if case["flow"] == "plume":  # the sweep's ranges
            nx, ny = int(r.integers(128, 513)), int(r.integers(64, 257))
            prm = dict(chi=r.uniform(0.1, 0.5), Dc=r.uniform(0.1, 0.3), gravity_scale=r.uniform(0.5, 2.0))
        else:  # the surrogate's parameter ranges
            nx = ny = case["n"]
            prm = dict(Ra=10 ** r.uniform(4, 6), Pr=0.7, Nc=r.uniform(-2, 2), Le=r.uniform(1, 10),
                       Sr=r.uniform(0, 0.5), Df=r.uniform(0, 0.5))
        pbs.append(_problem(case["flow"], nx, ny, prm))
    return pbs


def _batch_sizes_seed(case, seed):
    # the lattices' sizes belong to the sweep, not to the fields drawn for them
    return 17 if case["flow"] == "plume" else seed


# ---- the cases ------------------------------------------------------------------------
def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "lattice":
        pb = _problem(case["flow"], case["nx"], case["ny"])
        s = lib.Solver(pb, storage=case["storage"], init=False)
        f = _fields(case["flow"], case["nx"], case["ny"], gen)
        return dict(kind=kind, s=s, fields=f, out=torch.empty_like(f), steps=case["steps"])
    if kind == "lattice3d":
        s = lib.Solver3D(_problem3(case), init=False)
        return dict(kind=kind, s=s, fields=_fields3(case, seed), steps=case["steps"])
    if kind == "batch":
        pbs = _members(case, _batch_sizes_seed(case, seed))
        kw = dict(tile=(64, 4), mode=0) if case["flow"] == "cavity" else {}
        s = lib.BatchSolver(pbs, init=False, **kw)
        f = torch.cat([_fields(case["flow"], pb.nx, pb.ny, gen).reshape(-1) for pb in pbs])
        return dict(kind=kind, s=s, fields=f, out=torch.empty_like(f), steps=case["steps"])
    if kind == "unet":
        net = S.UNet(seed=seed)
        prm = S.draw_parameters(case["N"], seed)
        x = torch.as_tensor(S.input_planes(case["n"], prm)).cuda().to(torch.bfloat16)
        y = torch.rand((case["N"], case["n"], case["n"], S.OUT_PLANES), generator=gen, device="cuda") - 0.5
        return dict(kind=kind, net=net, x=x, y=y)
    shape = (case["N"], case["H"], case["W"])
    cin, cout = case["cin"], case["cout"]
    w = (torch.randn((cout, 3, 3, cin), generator=gen, device="cuda") * math.sqrt(2 / (9 * cin))).to(torch.bfloat16)
    # activations leave a ReLU: half of them are zero
    x = torch.randn(shape + (cin,), generator=gen, device="cuda").relu().to(torch.bfloat16)
    st = dict(kind=kind, w=w, x=x)
    if kind == "conv_fwd":
        st["b"] = 0.1 * torch.randn(cout, generator=gen, device="cuda")
    else:
        st["dy"] = torch.randn(shape + (cout,), generator=gen, device="cuda").to(torch.bfloat16)
    return st


def run(st):
    kind = st["kind"]
    if kind in ("lattice", "batch"):
        s = st["s"]
        s.init_moments_device(st["fields"])
        s.step(st["steps"])
        s.moments_device(st["out"])
        return st["out"]
    if kind == "lattice3d":
        s = st["s"]
        s.init_moments(*st["fields"])
        s.step(st["steps"])
        return s.moments()
    if kind == "conv_fwd":
        return S.conv3x3_fwd(st["x"], st["w"], st["b"], True)
    if kind == "conv_bwd":
        w, dy = st["w"], st["dy"]
        dw = torch.zeros(w.shape, dtype=torch.float32, device="cuda")
        db = torch.zeros(w.shape[0], dtype=torch.float32, device="cuda")
        S.conv3x3_bwd_weight(st["x"], dy, dw, db)
        return dict(dx=S.conv3x3_bwd_data(dy, w, w.shape[3]), dw=dw, db=db)
    out, acts = st["net"].forward(st["x"])
    loss, dout = S.mse(out, st["y"])
    return dict(out=out, loss=loss, grads=st["net"].backward(acts, dout))


def _unet_layers():
    """(lattice level, input channels, output channels) of the network's convolutions."""
    ch, prev, got = [32, 64, 128, 256], S.IN_PAD, []
    for lv, c in enumerate(ch):
        got += [(lv, prev, c), (lv, c, c)]
        prev = c
    for lv in (2, 1, 0):
        got += [(lv, ch[lv + 1] + ch[lv], ch[lv]), (lv, ch[lv], ch[lv])]
    return got


def _conv_work(P, cin, cout):
    return 2.0 * P * 9 * cin * cout


def work(case):
    kind = case["kind"]
    if kind in ("lattice", "lattice3d", "batch"):
        # moments in and out once; per node update the sums, equilibria and
        # relaxations of the model (counted on its equations for two scalars)
        if kind == "batch":
            nodes = sum(pb.nx * pb.ny for pb in _members(case, _batch_sizes_seed(case, 0)))
        else:
            nodes = case["nx"] * case["ny"] * case.get("nz", 1)
        per = 480 if kind == "lattice3d" else (150 if case["flow"] == "cellular" else 300)
        return dict(bytes=2.0 * (8 * (M + 4) if kind == "lattice3d" else 4 * (M + 3)) * nodes,
                    flops=float(per) * nodes * case["steps"])
    if kind == "unet":
        P = case["N"] * case["n"] ** 2
        flops = params = acts = 0.0
        for lv, cin, cout in _unet_layers():
            flops += 3 * _conv_work(P / 4 ** lv, cin, cout)
            params += 9.0 * cin * cout
            acts += 2.0 * P / 4 ** lv * cout  # each layer's output, kept for the backward pass
        return dict(bytes=P * (2.0 * S.IN_PAD + 8.0 * S.OUT_PLANES) + 2 * acts + 6 * params, flops=flops)
    P, cin, cout = case["N"] * case["H"] * case["W"], case["cin"], case["cout"]
    if kind == "conv_fwd":
        return dict(bytes=2.0 * P * (cin + cout) + 18.0 * cin * cout, flops=_conv_work(P, cin, cout))
    return dict(bytes=2.0 * P * (2 * cin + cout) + 54.0 * cin * cout, flops=2 * _conv_work(P, cin, cout))


# ---- the same in 64 bits --------------------------------------------------------------
def _velocities(dim):
    if dim == 2:
        c9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        return c9, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, c9[:5], [1 / 3] + [1 / 6] * 4, 1 / 3
    axes = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    diag = [tuple(c) for c in np.ndindex(3, 3, 3) if sum(k != 1 for k in c) == 2]
    diag = [tuple(k - 1 for k in c) for c in diag]
    c19 = [(0, 0, 0)] + axes + diag
    return c19, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, [(0, 0, 0)] + axes, [1 / 4] + [1 / 8] * 6, 1 / 4


def _lattice64(pb, fields, steps, sides, g):
    """The model on one lattice in 64 bits.  fields: phi, u (x first), p in arrays whose
    last axis is x; sides: low and high side of x, y(, z); returns phi, u, p stacked."""
    dim = len(sides) // 2
    cf, Wf, cs, Ws, cs2 = _velocities(dim)
    case1 = getattr(pb, "case1", False)
    phi, u, p = fields[:M], fields[M:M + dim], fields[M + dim]
    dev = phi.device
    axis = [phi.dim() - 2 - d for d in range(dim)]  # of one field, for x, y, z
    D = torch.as_tensor(pb.D, device=dev)
    beta, ref = [float(b) for b in pb.beta], [float(r) for r in pb.phi_ref]
    wf = 1 / (3 * pb.nu + 0.5)
    chem, consume = pb.dkind == "chemotaxis", pb.skind == "consumption"
    # which nodes a link c comes into from beyond a wall, and through which side
    edge = []
    for d in range(dim):
        for hi in (0, 1):
            m = torch.zeros(p.shape, dtype=torch.bool, device=dev)
            if sides[2 * d].kind == I.WALL:
                m.select(axis[d], -1 if hi else 0).fill_(True)
            edge.append(m)

    def crossed(c):
        return [2 * d + (0 if c[d] > 0 else 1) for d in range(dim) if c[d] != 0]

    def shifted(a, c):
        return torch.roll(a, [c[d] for d in range(dim)], [axis[d] for d in range(dim)])

    def dot(c, v):
        t = None
        for d in range(dim):
            if c[d]:
                t = c[d] * v[d] if t is None else t + c[d] * v[d]
        return 0.0 if t is None else t

    def closures(phi):
        r = (phi[1] >= pb.c_star).double() if chem or consume else None
        src = -pb.k * phi[0] * r if consume else None
        if chem:
            a, b = D[0, 0] / cs2 + 0.5, D[1, 1] / cs2 + 0.5
            o, q = D[0, 1] / cs2 - pb.chi / cs2 * phi[0] * r, D[1, 0] / cs2
            det = a * b - o * q
            om = [[b / det, -o / det], [-q / det, a / det]]
        else:
            inv = torch.linalg.inv(D / cs2 + 0.5 * torch.eye(M, device=dev, dtype=torch.float64))
            om = [[float(inv[i, j]) for j in range(M)] for i in range(M)]
        fm = pb.F0 + sum(beta[a] * (phi[a] - ref[a]) for a in range(M))
        return om, src, [float(g[d]) * fm for d in range(dim)]

    def collide(f, h, u, before, src_before):
        phi = [sum(f[a]) for a in range(M)]
        om, src, F = closures(phi)
        if case1:
            J = [[sum((float(a == b) - om[a][b] / 2) * u[d] * (phi[b] - before[b]) for b in range(M)) for d in range(dim)]
                 for a in range(M)]
            pr = torch.zeros_like(phi[0])
        else:
            u = [sum(c[d] * h[i] for i, c in enumerate(cf) if c[d]) + F[d] / 2 for d in range(dim)]
            uu = sum(v * v for v in u)
            pr = (sum(h[1:]) - Wf[0] * 1.5 * uu) / (3 * (1 - Wf[0]))
            S_ = [0.0, src if consume else 0.0]
            J = [[sum((float(a == b) - om[a][b] / 2) * (u[d] * S_[b] + phi[b] * F[d]) for b in range(M))
                  for d in range(dim)] for a in range(M)]
        new_f = [[None] * len(cs) for _ in range(M)]
        for i, c in enumerate(cs):
            neq = [f[b][i] - Ws[i] * phi[b] * (1 + dot(c, u) / cs2) for b in range(M)]
            for a in range(M):
                v = f[a][i] - sum(om[a][b] * neq[b] for b in range(M)) + Ws[i] * dot(c, J[a]) / cs2
                if a == 1 and consume:
                    v = v + Ws[i] * (1.5 * src - 0.5 * (src if src_before is None else src_before))
                new_f[a][i] = v
        new_h = h
        if not case1:
            new_h = [h[i] - wf * (h[i] - heq(i, pr, u, uu)) + (1 - wf / 2) * 3 * Wf[i] * dot(c, F)
                     for i, c in enumerate(cf)]
        return new_f, new_h, phi, u, pr, src

    def heq(i, pr, u, uu):
        if i == 0:
            return -3 * (1 - Wf[0]) * pr - 1.5 * Wf[0] * uu
        cu = dot(cf[i], u)
        return 3 * Wf[i] * (pr + cu + 1.5 * cu * cu - 0.5 * uu)

    def stream(f, h):
        nf = [[None] * len(cs) for _ in range(M)]
        for i, c in enumerate(cs):
            o = cs.index(tuple(-k for k in c))
            for a in range(M):
                v = shifted(f[a][i], c)
                for s in crossed(c):
                    wall = f[a][o]
                    if sides[s].kind == I.WALL and sides[s].scalar[a] == I.DIRICHLET:
                        wall = 2 * Ws[i] * sides[s].value[a] - wall
                    v = torch.where(edge[s], wall, v)
                nf[a][i] = v
        if case1:
            return nf, h
        nh = []
        for i, c in enumerate(cf):
            v = shifted(h[i], c)
            through = crossed(c)
            for s in through:
                v = torch.where(edge[s], h[cf.index(tuple(-k for k in c))], v)
            if dim == 2 and len(through) == 2:  # free slip: the mirrored link, except in corners
                for s, other in (through, through[::-1]):
                    if sides[s].kind == I.WALL and sides[s].fluid == I.FREESLIP:
                        d = s // 2
                        image = tuple(-k if e == d else k for e, k in enumerate(c))
                        along = tuple(0 if e == d else k for e, k in enumerate(c))
                        v = torch.where(edge[s] & ~edge[other], shifted(h[cf.index(image)], along), v)
            nh.append(v)
        return nf, nh

    u = [u[d] for d in range(dim)]
    f = [[Ws[i] * phi[a] * (1 + dot(c, u) / cs2) for i, c in enumerate(cs)] for a in range(M)]
    _, _, F = closures([phi[a] for a in range(M)])
    uu = sum(v * v for v in u)
    h = None if case1 else [heq(i, p, u, uu) - 1.5 * Wf[i] * dot(c, F) for i, c in enumerate(cf)]
    f, h, phi, u, pr, src = collide(f, h, u, [phi[a] for a in range(M)], None)
    for _ in range(steps):
        f, h = stream(f, h)
        f, h, phi, u, pr, src = collide(f, h, u, phi, src)
    return torch.stack(list(phi) + list(u) + [pr])


def _conv64(x, w, b=None):
    y = Fn.conv2d(x.permute(0, 3, 1, 2), w.permute(0, 3, 1, 2), b, padding=1)
    return y.permute(0, 2, 3, 1)


def _unet64(st):
    net = st["net"]
    P = {k: (net.bf16[k] if k in net.bf16 else t).double().requires_grad_(True) for k, t in net.master.items()}
    conv = lambda h, k: _conv64(h, P[k + ".w"], P[k + ".b"]).relu()  # noqa: E731
    h, skips = st["x"].double(), []
    for lv in range(net.levels):
        if lv:
            h = Fn.avg_pool2d(h.permute(0, 3, 1, 2), 2).permute(0, 2, 3, 1)
        h = conv(conv(h, f"e{lv}a"), f"e{lv}b")
        skips.append(h)
    for lv in range(net.levels - 2, -1, -1):
        h = torch.cat([h.repeat_interleave(2, 1).repeat_interleave(2, 2), skips[lv]], 3)
        h = conv(conv(h, f"d{lv}a"), f"d{lv}b")
    out = h @ P["head.w"].T + P["head.b"]
    loss = ((out - st["y"].double()) ** 2).mean()
    loss.backward()
    return dict(out=out.detach(), loss=loss.detach().reshape(1), grads={k: t.grad for k, t in P.items()})


def exact(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "lattice":
        pb = _problem(case["flow"], case["nx"], case["ny"])
        f = _fields(case["flow"], case["nx"], case["ny"], gen).double()
        return _lattice64(pb, f, case["steps"], [pb.west, pb.east, pb.south, pb.north], pb.g)
    if kind == "lattice3d":
        phi, u, p = (torch.as_tensor(a, device="cuda") for a in _fields3(case, seed))
        pb = _problem3(case)
        return _lattice64(pb, torch.cat([phi, u, p[None]]), case["steps"], pb.sides, pb.g).cpu().numpy()
    if kind == "batch":
        pbs = _members(case, _batch_sizes_seed(case, seed))
        if len(pbs) * case["steps"] > 4500:  # more small launches than 20 seconds hold
            return None
        return torch.cat([_lattice64(pb, _fields(case["flow"], pb.nx, pb.ny, gen).double(), case["steps"],
                                     [pb.west, pb.east, pb.south, pb.north], pb.g).reshape(-1) for pb in pbs])
    st = prepare(case, seed)
    if kind == "unet":
        return _unet64(st)
    x, w = st["x"].double(), st["w"].double()
    if kind == "conv_fwd":
        return _conv64(x, w, st["b"].double()).relu()
    dy = st["dy"].double().permute(0, 3, 1, 2)
    xs, ws = x.permute(0, 3, 1, 2), w.permute(0, 3, 1, 2)
    dx = torch.nn.grad.conv2d_input(xs.shape, ws, dy, padding=1).permute(0, 2, 3, 1)
    dw = torch.nn.grad.conv2d_weight(xs, ws.shape, dy, padding=1).permute(0, 2, 3, 1)
    return dict(dx=dx, dw=dw, db=dy.sum((0, 2, 3)))
