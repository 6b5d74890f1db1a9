"""The work a user of this package has it do, as cases to be timed and compared.

Each case is one pass through the public entry points: a run of time steps with the fields read
afterwards (one geometry or a batch), the warm-start network's prediction and training step, and one
of its convolution layers.  ``listed()`` names the cases, ``draw()`` takes one more from the same
ranges, ``prepare()`` makes the inputs and the handle a program keeps, ``run()`` is the pass,
``work()`` its unavoidable bytes and operations, ``exact()`` its results in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_1703_08015_gb300 import lbm, nn

STORAGE = {"f64": lbm.LBM_STORE_F64, "f32": lbm.LBM_STORE_F32, "f16s": lbm.LBM_STORE_F16S, "f32s": lbm.LBM_STORE_F32S}
WIDTH = {"f64": 8, "f32": 4, "f16s": 2, "f32s": 4}
ARITH = {"auto": lbm.LBM_ARITH_AUTO, "table": lbm.LBM_ARITH_FF_TABLE, "fixed": lbm.LBM_ARITH_FIXED,
         "native": lbm.LBM_ARITH_F64}
MODEL = {"quasi": lbm.LBM_QUASI_COMPRESSIBLE, "incompressible": lbm.LBM_INCOMPRESSIBLE}
LAYOUT = {"t2c": lbm.LBM_LAYOUT_T2C, "tgb": lbm.LBM_LAYOUT_TGB}
FORCE = 1e-6


def _flow(name, geometry, nx, ny, nz, fluid, storage="f64", tile=4, steps=20, check=False, arith="auto",
          model="quasi", layout="t2c", tau=0.6):
    c = dict(kind="flow", geometry=geometry, nx=nx, ny=ny, nz=nz, fluid=fluid, storage=storage, tile=tile,
             steps=steps, check=check, arith=arith, model=model, layout=layout, tau=tau)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a 2D microchannel chip between two reads of its fields: the smallest domain, all latency
        _flow("circles_2d_128_f64", "circles", 128, 128, 1, 0.5, tile=16, steps=100, tau=0.8),
        # one residual check of a steady-state solve on a 64^3 rock sample (what time-to-steady repeats),
        # in the double-precision form and in the reduced form that most solves use
        _flow("pack_64_f64_check", "spheres", 64, 64, 64, 0.35, steps=100, check=True),
        _flow("pack_64_f32s_check", "spheres", 64, 64, 64, 0.35, storage="f32s", steps=100, check=True),
        # a rock sample in double precision, the size of a production run
        _flow("pack_256_f64", "spheres", 256, 256, 256, 0.3),
        # a vessel tree: 5 % fluid in a large box, single precision
        _flow("tubes_256_f32", "tubes", 256, 256, 256, 0.05, storage="f32"),
        # the same rock in half-precision deviations
        _flow("pack_256_f16s", "spheres", 256, 256, 256, 0.3, storage="f16s"),
        # a scanned sample whose sides are no multiples of the tile
        _flow("pack_ragged_f32s", "spheres", 192, 177, 203, 0.35, storage="f32s"),
        # one copy updated in place (half the memory)
        _flow("pack_128_f64_in_place", "spheres", 128, 128, 128, 0.3, layout="tgb"),
        # 64 samples of uneven size and porosity in one launch per step: a residual check of the
        # training-data production, and every sample's fields
        dict(name="batch_64_f32s", kind="batch", samples=64, side_min=32, side_max=160, storage="f32s", steps=20),
        # warm-start prediction for one geometry
        dict(name="predict_64", kind="predict", n=1, d=64, h=64, w=64),
        # one training step of the network
        dict(name="train_64_batch8", kind="train", n=8, d=64, h=64, w=64),
        # one convolution layer, forward and backward (the decoder's widest input)
        dict(name="conv_96_32", kind="conv", n=8, d=32, h=32, w=32, cin=96, cout=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow2d", "flow3d", "flow3d", "flow3d", "batch", "predict", "train", "conv", "conv"])
    if kind == "flow2d":
        tile = rng.choice([8, 16, 32])
        return _flow(None, "circles", tile * max(1, _log_int(rng, 48, 1000) // tile), _log_int(rng, 40, 1000), 1,
                     round(rng.uniform(0.3, 0.8), 3), storage=rng.choice(["f64", "f64", "f32s", "f32"]), tile=tile,
                     steps=_log_int(rng, 1, 100), check=rng.random() < 0.3,
                     model=rng.choice(["quasi", "incompressible"]), tau=round(rng.uniform(0.55, 1.2), 3))
    if kind == "flow3d":
        tile = rng.choice([4, 4, 4, 8])
        nx = tile * max(1, _log_int(rng, 24, 224) // tile)
        ny, nz = _log_int(rng, 24, 224), _log_int(rng, 24, 224)
        storage = rng.choice(["f64", "f64", "f32s", "f32s", "f32", "f16s"])
        layout = "tgb" if rng.random() < 0.15 else "t2c"
        arith = rng.choice(["auto", "auto", "auto", "auto", "table", "fixed", "native"]) if storage == "f64" else "auto"
        steps = min(_log_int(rng, 1, 100), max(1, 200_000_000 // (nx * ny * nz)))
        return _flow(None, rng.choice(["spheres", "spheres", "tubes"]), nx, ny, nz, round(rng.uniform(0.05, 0.6), 3),
                     storage=storage, tile=tile, steps=steps, check=layout == "t2c" and rng.random() < 0.4,
                     arith=arith, model=rng.choice(["quasi", "quasi", "incompressible"]), layout=layout,
                     tau=round(rng.uniform(0.55, 1.0), 3))
    if kind == "batch":
        return dict(kind="batch", samples=_log_int(rng, 2, 64), side_min=32, side_max=8 * rng.randrange(5, 17),
                    storage=rng.choice(["f32s", "f32s", "f64"]), steps=_log_int(rng, 2, 20))
    if kind in ("predict", "train"):
        return dict(kind=kind, n=rng.randrange(1, 9 if kind == "train" else 5),
                    **{a: 8 * rng.randrange(2, 9) for a in ("d", "h", "w")})
    return dict(kind="conv", n=rng.randrange(1, 9), d=rng.randrange(6, 49), h=rng.randrange(6, 49),
                w=rng.randrange(6, 49), cin=rng.choice([2, 16, 32, 48, 64, 96, 128, 192]),
                cout=rng.choice([4, 16, 32, 64, 128]))


# ---- geometries ------------------------------------------------------------------------------


def _spheres(shape, fluid, rng, r_min=4.0, r_max=12.0):
    """Overlapping solid spheres (discs for nz = 1) of uniform radius, periodic along x: [z][y][x], 1 = fluid."""
    nz, ny, nx = shape
    d3 = nz > 1
    mean = (4.0 / 3.0 * math.pi * (r_max ** 4 - r_min ** 4) / 4.0 if d3
            else math.pi * (r_max ** 3 - r_min ** 3) / 3.0) / (r_max - r_min)
    # spheres also centred outside the walls, so that the porosity is the same up to them
    pad = r_max if d3 else 0.0
    box = nx * (ny + 2 * r_max) * (nz + 2 * pad)
    count = max(1, int(round(-math.log(fluid) * box / mean)))
    c = rng.uniform((0.0, -r_max, -pad), (nx, ny + r_max, nz + pad if d3 else 1e-9), (count, 3))
    r = rng.uniform(r_min, r_max, count)
    solid = torch.zeros((nz, ny, nx), dtype=torch.bool, device="cuda")
    k = int(math.ceil(r_max)) + 1
    span = torch.arange(-k, k + 1, device="cuda")
    dz, dy, dx = torch.meshgrid(span if d3 else span[:1] * 0, span, span, indexing="ij")
    off = torch.stack([dx.reshape(-1), dy.reshape(-1), dz.reshape(-1)], 1)
    c, r = torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda()
    for b in range(0, count, 512):
        at = c[b:b + 512].floor().long()[:, None, :] + off[None]
        inside = ((at - c[b:b + 512, None, :]) ** 2).sum(2) <= (r[b:b + 512] ** 2)[:, None]
        x, y, z = at[..., 0] % nx, at[..., 1], at[..., 2]
        inside &= (y >= 0) & (y < ny) & (z >= 0) & (z < nz)
        solid[z[inside], y[inside], x[inside]] = True
    return (~solid).to(torch.uint8)


def _tubes(shape, fluid, rng, r_min=3.0, r_max=10.0):
    """Straight tubes of uniform radius in solid rock, half of them along x, until the fluid fraction is reached."""
    nz, ny, nx = shape
    open_ = torch.zeros(shape, dtype=torch.bool, device="cuda")
    z, y, x = (torch.arange(n, device="cuda", dtype=torch.float32) for n in shape)
    for _ in range(400):
        r = rng.uniform(r_min, r_max)
        p = rng.uniform((0.0, 0.0, 0.0), (nx, ny, nz))
        v = rng.normal(size=3)
        v = np.array([1.0, 0.0, 0.0]) if rng.random() < 0.5 else v / np.linalg.norm(v)
        ex, ey, ez = x[None, None, :] - p[0], y[None, :, None] - p[1], z[:, None, None] - p[2]
        t = ex * v[0] + ey * v[1] + ez * v[2]
        open_ |= ex * ex + ey * ey + ez * ez - t * t <= r * r
        if float(open_.float().mean()) >= fluid:
            break
    return open_.to(torch.uint8)


def _mask(geometry, shape, fluid, rng):
    """A geometry in host memory, as lbm_init takes it."""
    if geometry == "tubes":
        m = _tubes(shape, fluid, rng)
    elif geometry == "circles":
        m = _spheres(shape, fluid, rng, 3.0, 8.0)
    else:
        m = _spheres(shape, fluid, rng)
    m[shape[0] // 2, shape[1] // 2, :] = 1  # never a box without any fluid
    return m.cpu().numpy()


def _start_fields(shape, dims, rng):
    """A smooth density and a velocity as a warm start gives them, FP64 on the device."""
    nz, ny, nx = shape
    g = torch.meshgrid(*(torch.arange(n, device="cuda", dtype=torch.float64) / n for n in shape), indexing="ij")

    def wave(size):
        f = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for _ in range(3):
            k = rng.integers(1, 4, 3)
            f += rng.normal() * torch.sin(2 * math.pi * (k[0] * g[0] + k[1] * g[1] + k[2] * g[2] + rng.random()))
        return size * f

    rho = 1.0 + wave(1e-4)
    return rho, torch.stack([wave(1e-3) for _ in range(dims)])


# ---- preparing and running ---------------------------------------------------------------------


def _flow_inputs(case, seed):
    rng = np.random.default_rng(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    mask = _mask(case["geometry"], shape, case["fluid"], rng)
    dims = 2 if case["geometry"] == "circles" else 3
    return mask, _start_fields(shape, dims, rng)


def _batch_sides(case):
    """The samples' sides, multiples of 8: the case's own, whatever the seed."""
    rng = np.random.default_rng(case["samples"])
    return [8 * int(k) for k in rng.integers(case["side_min"] // 8, case["side_max"] // 8 + 1, case["samples"])]


def _batch_masks(case, seed):
    rng = np.random.default_rng(seed)
    masks = []
    for side in _batch_sides(case):
        masks.append(_mask("spheres", (side,) * 3, float(rng.uniform(0.1, 0.6)), rng))
    return masks


def _net_inputs(case, seed):
    rng = np.random.default_rng(seed)
    shape = (case["d"], case["h"], case["w"])
    masks = np.stack([_mask("spheres", shape, float(rng.uniform(0.1, 0.6)), rng) for _ in range(case["n"])])
    target = torch.stack([torch.stack([f * 1e3 for f in _start_fields(shape, 3, rng)[1]] * 2)[:4].movedim(0, -1)
                          for _ in range(case["n"])]).float()
    m = torch.from_numpy(masks).cuda()
    return m, target * m[..., None]


def _train_state(case, seed):
    """A network in the middle of its training: weights and the optimiser's moments."""
    net = nn.UNet(seed=seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    net.m.copy_(1e-3 * torch.randn(net.n_params, device="cuda", generator=g))
    net.v.copy_(1e-4 * (0.5 + torch.rand(net.n_params, device="cuda", generator=g)))
    net.t = 1000
    return net


def _conv_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(scale, *size):
        return (scale * torch.randn(*size, device="cuda", generator=g)).to(torch.bfloat16)

    vox = (case["n"], case["d"], case["h"], case["w"])
    x = torch.relu(normal(1.0, *vox, case["cin"]))
    w = normal(math.sqrt(2.0 / (27 * case["cin"])), 27, case["cin"], case["cout"])
    b = 0.1 * torch.randn(case["cout"], device="cuda", generator=g)
    return x, w, b, normal(1e-2, *vox, case["cout"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "flow":
        mask, (rho, u) = _flow_inputs(case, seed)
        d2 = case["geometry"] == "circles"
        s = lbm.Solver(mask, lbm.LBM_D2Q9 if d2 else lbm.LBM_D3Q19, case["tile"], (1, 0, 0), case["tau"],
                       (FORCE, 0.0, 0.0), model=MODEL[case["model"]], storage=STORAGE[case["storage"]],
                       arith=ARITH[case["arith"]], rho_init=rho, u_init=u, layout=LAYOUT[case["layout"]])
        if case["check"]:
            s.stats(residual=True)
        return dict(case=case, solver=s, rho=torch.empty_like(rho), u=torch.empty_like(u))
    if kind == "batch":
        masks = _batch_masks(case, seed)
        b = lbm.BatchSolver(masks, lbm.LBM_D3Q19, 4, (1, 0, 0), 0.6, (FORCE, 0.0, 0.0),
                            storage=STORAGE[case["storage"]])
        b.stats(residual=True)
        total = sum(m.size for m in masks)
        rho = torch.empty(total, dtype=torch.float64, device="cuda")
        u = torch.empty(3 * total, dtype=torch.float64, device="cuda")
        at = np.cumsum([0] + [m.size for m in masks])
        parts = [(rho[at[k]:at[k + 1]], u[3 * at[k]:3 * at[k + 1]]) for k in range(len(masks))]
        return dict(case=case, solver=b, rho=rho, u=u, parts=parts)
    if kind == "predict":
        return dict(case=case, net=nn.UNet.load(nn.WEIGHTS), mask=_net_inputs(case, seed)[0])
    if kind == "train":
        mask, target = _net_inputs(case, seed)
        net = _train_state(case, seed)
        return dict(case=case, net=net, x=nn.inputs_from_masks(mask, FORCE, net._s()), mask=mask, target=target,
                    count=int(mask.sum()), loss=torch.zeros(1, dtype=torch.float64, device="cuda"))
    x, w, b, dy = _conv_inputs(case, seed)
    return dict(case=case, x=x, w=w, b=b, dy=dy)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "flow":
        s = state["solver"]
        s.step(case["steps"])
        out = dict(rho=state["rho"], u=state["u"])
        if case["check"]:
            st, _ = s.stats(residual=True)
            out["stats"] = np.array([st.mass, st.momentum[0], st.u2])
            out["n_fluid"] = int(st.n_fluid)
            s.filter_period2()
        lbm.lbm_moments(s.ctx, state["rho"], state["u"], None, lbm.LBM_OUT_DEVICE, s._s())
        return out
    if kind == "batch":
        b = state["solver"]
        b.step(case["steps"])
        stats, _ = b.stats(residual=True)
        b.filter_period2()
        for k, (rho, u) in enumerate(state["parts"]):
            lbm.lbm_moments_sample(b.ctx, k, rho, u, lbm.LBM_OUT_DEVICE, b._s())
        return dict(rho=state["rho"], u=state["u"],
                    stats=np.array([[st.mass, st.momentum[0], st.u2] for st in stats]),
                    n_fluid=np.array([st.n_fluid for st in stats]))
    if kind == "predict":
        net, m = state["net"], state["mask"]
        return net.forward(nn.inputs_from_masks(m, FORCE, net._s()), tuple(m.shape))
    if kind == "train":
        net, t = state["net"], state["target"]
        y = net.forward(state["x"], tuple(state["mask"].shape), keep=True)
        dout = torch.empty(y.shape, dtype=torch.bfloat16, device=y.device)
        nn.lbm_nn_mse(y, t, state["mask"], state["mask"].numel(), net.cout, state["count"], state["loss"], dout, net._s())
        net.backward(dout)
        net.adam(1e-3)
        return dict(p=net.p, m=net.m, v=net.v)
    x, w, b, dy = state["x"], state["w"], state["b"], state["dy"]
    dims, cin, cout = tuple(x.shape[:4]), x.shape[4], w.shape[2]
    y, y32 = torch.empty_like(dy), torch.empty(dy.shape, device="cuda")
    dx, wt = torch.empty_like(x), torch.empty_like(w)
    dw, db = torch.zeros(w.shape, device="cuda"), torch.zeros(cout, device="cuda")
    nn.lbm_nn_conv3d(x, *dims, cin, w, b, cout, 1, 1, y, y32)
    nn.lbm_nn_weight_flip(w, cin, cout, wt)
    nn.lbm_nn_conv3d_wgrad(x, dy, *dims, cin, cout, 1, dw, db)
    nn.lbm_nn_conv3d(dy, *dims, cout, wt, None, cin, 0, 1, dx, None)
    return dict(y=y, y32=y32, dx=dx, dw=dw, db=db)


# ---- what a pass cannot do without ---------------------------------------------------------------


def work(case):
    kind = case["kind"]
    if kind in ("flow", "batch"):
        if kind == "flow":
            boxes, fluid = [case["nx"] * case["ny"] * case["nz"]], case["fluid"]
            q, d = (9, 2) if case["geometry"] == "circles" else (19, 3)
        else:
            boxes, fluid, q, d = [s ** 3 for s in _batch_sides(case)], 0.35, 19, 3
        nodes = sum(boxes) * fluid
        passes = 2 * case["steps"] + 1  # every step reads and writes the state; the fields read it once more
        if case.get("check") or kind == "batch":
            passes += 4  # the residual's sums read it, the filter reads two states and writes one
        return dict(bytes=nodes * q * WIDTH[case["storage"]] * passes + sum(boxes) * 8 * (1 + d),
                    flops=nodes * case["steps"] * 13 * q)
    vox = case["n"] * case["d"] * case["h"] * case["w"]
    if kind == "conv":
        one = 2 * 27 * case["cin"] * case["cout"] * vox
        return dict(bytes=vox * (4 * case["cin"] + 8 * case["cout"]) + 27 * 8 * case["cin"] * case["cout"],
                    flops=3 * one)
    flops, params = 0, 0
    for name, ci, co, _ in nn.unet_layers((16, 32, 64, 128), 2, 4):
        level = 3 if name.startswith("mid") else (int(name[3]) if name[:3] in ("enc", "dec") else 0)
        flops += 2 * 27 * ci * co * vox / 8 ** level
        params += 27 * ci * co + co
    if kind == "predict":
        return dict(bytes=vox * (1 + 16) + 2 * params, flops=flops)
    return dict(bytes=vox * (4 + 1 + 16) + params * 4 * 6, flops=3 * flops)


# ---- the same results in plain 64-bit torch ---------------------------------------------------------

D2Q9_C = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
D3Q19_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
           (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
           (0, -1, 1)]


class _Lattice:
    """BGK on the dense masked box, periodic along x, halfway bounce-back elsewhere, Guo forcing along x."""

    def __init__(self, mask, two_d, tau, incompressible):
        self.c = D2Q9_C if two_d else D3Q19_C
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if two_d else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        self.w = [w[sum(map(abs, c))] for c in self.c]
        self.opp = [self.c.index((-c[0], -c[1], -c[2])) for c in self.c]
        self.tau, self.inc = tau, incompressible
        self.fluid = torch.from_numpy(mask).cuda().bool()
        self.from_fluid = [self.pull(self.fluid, c) for c in self.c]

    @staticmethod
    def pull(a, c):
        """a(r - c): wrapped along x, zero beyond the other walls."""
        a = torch.roll(a, c[0], 2) if c[0] else a
        for axis, s in ((1, c[1]), (0, c[2])):
            if s:
                a = torch.roll(a, s, axis)
                a.select(axis, 0 if s > 0 else a.shape[axis] - 1).zero_()
        return a

    def equilibrium(self, i, rho, u, usq):
        cu = sum(self.c[i][k] * u[k] for k in range(3) if self.c[i][k]) if i else torch.zeros_like(rho)
        poly = 3 * cu + 4.5 * cu * cu - 1.5 * usq
        return self.w[i] * (rho + poly if self.inc else rho * (1 + poly)), cu

    def start(self, rho, u):
        u = [u[k] if k < len(u) else torch.zeros_like(rho) for k in range(3)]
        usq = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        self.f = [self.equilibrium(i, rho, u, usq)[0] for i in range(len(self.c))]
        self.last = None

    def gathered(self, f):
        return [torch.where(self.from_fluid[i], self.pull(f[i], self.c[i]), f[self.opp[i]])
                for i in range(len(self.c))]

    def moments(self, g):
        rho = sum(g)
        j = [sum(self.c[i][k] * g[i] for i in range(len(g)) if self.c[i][k]) for k in range(3)]
        j = [torch.zeros_like(rho) if isinstance(v, int) else v for v in j]
        j[0] = j[0] + 0.5 * FORCE
        return rho, (j if self.inc else [v / rho for v in j])

    def step(self):
        g = self.gathered(self.f)
        rho, u = self.moments(g)
        usq, om = u[0] ** 2 + u[1] ** 2 + u[2] ** 2, 1.0 / self.tau
        out = []
        for i in range(len(g)):
            feq, cu = self.equilibrium(i, rho, u, usq)
            s = (1 - 0.5 * om) * self.w[i] * FORCE * (3 * (self.c[i][0] - u[0]) + 9 * cu * self.c[i][0])
            out.append(g[i] - om * (g[i] - feq) + s)
        self.last, self.f = self.f, out

    def fields(self):
        rho, u = self.moments(self.gathered(self.f))
        nan = torch.full_like(rho, float("nan"))
        return torch.where(self.fluid, rho, nan), [torch.where(self.fluid, v, nan) for v in u]

    def stats(self):
        rho, u = self.moments(self.gathered(self.f))
        rho, u = rho[self.fluid], [v[self.fluid] for v in u]
        px = (rho * u[0]).sum()
        return np.array([float(rho.sum()), float(px), float(u[0].square().sum() + u[1].square().sum() + u[2].square().sum())])

    def filter_period2(self):
        self.f = [0.5 * (a + b) for a, b in zip(self.f, self.last)]


def _solve(mask, two_d, tau, incompressible, start, steps, check):
    lat = _Lattice(mask, two_d, tau, incompressible)
    lat.start(*start)
    for _ in range(steps):
        lat.step()
    stats = None
    if check:
        stats = lat.stats()
        lat.filter_period2()
    rho, u = lat.fields()
    return rho, torch.stack(u[:2 if two_d else 3]), stats, int(lat.fluid.sum())


def _conv64(x, w, b=None, relu=False):
    """3x3x3, zero padding, periodic along x: float64 [n][z][y][x][c] by [27][cin][cout]."""
    n, d, h, wd, ci = x.shape
    p = torch.zeros((n, d + 2, h + 2, wd + 2, ci), dtype=torch.float64, device="cuda")
    p[:, 1:-1, 1:-1, 1:-1] = x
    p[:, 1:-1, 1:-1, 0], p[:, 1:-1, 1:-1, -1] = x[..., -1, :], x[..., 0, :]
    y = torch.zeros((n, d, h, wd, w.shape[2]), dtype=torch.float64, device="cuda")
    for t in range(27):
        z, yy, xx = t // 9, t // 3 % 3, t % 3
        y += p[:, z:z + d, yy:yy + h, xx:xx + wd] @ w[t]
    if b is not None:
        y = y + b
    return torch.relu(y) if relu else y


def _wgrad64(x, dy):
    n, d, h, wd, ci = x.shape
    p = torch.zeros((n, d + 2, h + 2, wd + 2, ci), dtype=torch.float64, device="cuda")
    p[:, 1:-1, 1:-1, 1:-1] = x
    p[:, 1:-1, 1:-1, 0], p[:, 1:-1, 1:-1, -1] = x[..., -1, :], x[..., 0, :]
    g = dy.reshape(-1, dy.shape[-1])
    dw = torch.stack([p[:, t // 9:t // 9 + d, t // 3 % 3:t // 3 % 3 + h, t % 3:t % 3 + wd].reshape(-1, ci).T @ g
                      for t in range(27)])
    return dw, g.sum(0)


def _flip(w):
    return w.flip(0).transpose(1, 2).contiguous()


def _bf(x):
    """What a BF16 tensor keeps of 64-bit values."""
    return x.float().to(torch.bfloat16).double()


def _blocks8(x):
    n, d, h, w, c = x.shape
    return x.reshape(n, d // 2, 2, h // 2, 2, w // 2, 2, c).sum((2, 4, 6))


def _up(x):
    return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)


def _net64(net, x, dout=None):
    """The U-Net with BF16 activations and weights and 64-bit sums; with `dout` (a function of the output)
    the parameter gradients as one flat vector."""
    P = {L.name: (_bf(net.p[L.w_off:L.w_off + L.nw].double()).view(27, L.cin, L.cout),
                  net.p[L.b_off:L.b_off + L.cout].double(), L) for L in net.layers}
    ins, outs = {}, {}

    def conv(name, a):
        w, b, L = P[name]
        ins[name] = a
        y = _conv64(a, w, b, L.relu)
        outs[name] = y if name == "head" else _bf(y)
        return outs[name]

    nl = len(net.chans) - 1
    a = x.double()
    for lv in range(nl):
        a = _bf(0.125 * _blocks8(conv(f"enc{lv}b", conv(f"enc{lv}a", a))))
    a = conv("mid_b", conv("mid_a", a))
    for lv in reversed(range(nl)):
        a = conv(f"dec{lv}b", conv(f"dec{lv}a", torch.cat([_up(a), outs[f"enc{lv}b"]], -1)))
    y = conv("head", a)
    if dout is None:
        return y
    grad = torch.zeros(net.n_params, dtype=torch.float64, device="cuda")

    def back(name, g, need_dx=True):
        w, _, L = P[name]
        if L.relu:
            g = torch.where(outs[name] > 0, g, torch.zeros_like(g))
        dw, db = _wgrad64(ins[name], g)
        grad[L.w_off:L.w_off + L.nw] = dw.reshape(-1)
        grad[L.b_off:L.b_off + L.cout] = db
        return _bf(_conv64(g, _flip(w))) if need_dx else None

    g, dskip = back("head", dout(y)), {}
    for lv in range(nl):
        g = back(f"dec{lv}a", back(f"dec{lv}b", g))
        c = net.chans[lv + 1]
        dskip[lv], g = g[..., c:], _bf(_blocks8(g[..., :c]))
    g = back("mid_a", back("mid_b", g))
    for lv in reversed(range(nl)):
        g = _bf(_bf(0.125 * _up(g)) + dskip[lv])
        g = back(f"enc{lv}a", back(f"enc{lv}b", g), lv > 0)
    return grad


def exact(case, seed):
    kind = case["kind"]
    if kind == "flow":
        mask, start = _flow_inputs(case, seed)
        rho, u, stats, n = _solve(mask, case["geometry"] == "circles", case["tau"], case["model"] == "incompressible",
                                  start, case["steps"], case["check"])
        out = dict(rho=rho, u=u)
        return dict(out, stats=stats, n_fluid=n) if case["check"] else out
    if kind == "batch":
        got = []
        for m in _batch_masks(case, seed):
            rest = (torch.ones(m.shape, dtype=torch.float64, device="cuda"),
                    torch.zeros((3,) + m.shape, dtype=torch.float64, device="cuda"))
            got.append(_solve(m, False, 0.6, False, rest, case["steps"], True))
        return dict(rho=torch.cat([g[0].reshape(-1) for g in got]), u=torch.cat([g[1].reshape(-1) for g in got]),
                    stats=np.array([g[2] for g in got]), n_fluid=np.array([g[3] for g in got]))
    if kind == "predict":
        net = nn.UNet.load(nn.WEIGHTS)
        m = _net_inputs(case, seed)[0].double()
        return _net64(net, torch.stack([m, torch.full_like(m, FORCE / nn.FORCE_REF)], -1))
    if kind == "train":
        mask, target = _net_inputs(case, seed)
        net, m = _train_state(case, seed), mask.double()
        x = torch.stack([m, torch.full_like(m, FORCE / nn.FORCE_REF)], -1)
        scale = 2.0 / (int(mask.sum()) * net.cout)
        g = _net64(net, x, lambda y: _bf(scale * (y - target.double()) * m[..., None]))
        b1, b2, lr, eps, t = 0.9, 0.999, 1e-3, 1e-8, net.t + 1
        mm = b1 * net.m.double() + (1 - b1) * g
        vv = b2 * net.v.double() + (1 - b2) * g * g
        p = net.p.double() - lr * mm / (1 - b1 ** t) / ((vv / (1 - b2 ** t)).sqrt() + eps)
        return dict(p=p, m=mm, v=vv)
    x, w, b, dy = _conv_inputs(case, seed)
    x64, w64, dy64 = x.double(), w.double(), dy.double()
    y = _conv64(x64, w64, b.double(), True)
    dw, db = _wgrad64(x64, dy64)
    return dict(y=y, y32=y, dx=_conv64(dy64, _flip(w64)), dw=dw, db=db)
