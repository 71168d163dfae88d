"""Timed workloads of the library, through its public entry points.

A case is a dict of plain values.  `listed` gives the fixed ones, `draw` more
of the same ranges, `prepare` what a program holds before the call, `run` one
pass, `work` the bytes and operations of a pass that cannot be avoided, and
`exact` what `run` returns for a fresh state, computed in 64 bits with plain
torch from the definitions of the method and the network.

Kinds:
  cavity    steps of one cavity, then its residual, hot-wall Nusselt numbers
            and fields: the monitoring loop of every solve
  ensemble  steps of a batch of cavities, residuals, Nusselt numbers, fields
            of all members: the generation of training data
  conv      one 3^3 convolution layer of the warm-start network
  predict   the network's prediction of steady states
  gradients loss and parameter gradients of a training batch
"""

import math
import os

import numpy as np
import torch

from paper_1511_04633_gb300 import dmrt, surrogate

PR, MA, INTERVAL = 0.71, 0.1, 100
STORAGES = {"f32": dmrt.STORE_F32, "bf16": dmrt.STORE_BF16, "f16": dmrt.STORE_F16}
STREAMINGS = {"two": dmrt.STREAM_AB, "inplace": dmrt.STREAM_INPLACE}
NETS = {"unet64": (64, 3, (16, 32, 64, 128)), "unet32": (32, 2, (16, 32, 64))}
BIGGEST = 256 ** 3 * 100  # cell updates of the largest listed cavity


def _cavity(name, grid, wall, ra, storage, streaming, steps):
    return {"name": name, "kind": "cavity", "nx": grid[0], "ny": grid[1], "nz": grid[2], "wall": wall, "ra": ra,
            "storage": storage, "streaming": streaming, "steps": steps}


def listed():
    return [
        # a few steps of a small box between two looks at it
        _cavity("tiny_f32_10", (16, 16, 16), 1, 1e4, "f32", "two", 10),
        # the validation cavity, one residual interval
        _cavity("cube32_f32", (32, 32, 32), 1, 1e3, "f32", "two", 100),
        # the paper's table grid, two intervals (so a residual exists)
        _cavity("cube60_f32_inplace", (60, 60, 60), 3, 1e5, "f32", "inplace", 200),
        # the benchmark cavity
        _cavity("cube128_f32", (128, 128, 128), 2, 1e5, "f32", "two", 100),
        # odd rows: an arbitrary box a user meshes, half the memory
        _cavity("odd_f16_inplace", (101, 75, 61), 1, 5e5, "f16", "inplace", 100),
        # even rows, nothing a multiple of anything, 16-bit
        _cavity("ragged_bf16", (190, 126, 90), 2, 3e5, "bf16", "two", 150),
        # the large reduced-storage cavity
        _cavity("cube256_bf16", (256, 256, 256), 3, 1e6, "bf16", "two", 100),
        # the 64-member batch of mixed cubes that makes training data
        {"name": "ensemble64_bf16", "kind": "ensemble", "count": 64, "edges": "32,48,64,96", "storage": "bf16",
         "streaming": "two", "steps": 100},
        # first level of the network at the training batch
        {"name": "conv_64_16_16", "kind": "conv", "n": 64, "batch": 4, "cin": 16, "cout": 16},
        # a deep level of the network
        {"name": "conv_16_64_64", "kind": "conv", "n": 16, "batch": 4, "cin": 64, "cout": 64},
        # one warm start's prediction
        {"name": "predict_64", "kind": "predict", "net": "unet64", "batch": 1},
        # one training batch
        {"name": "gradients_64", "kind": "gradients", "net": "unet64", "batch": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cavity"] * 5 + ["ensemble", "conv", "conv", "predict", "gradients"])
    if kind == "cavity":
        while True:
            grid = [_log_int(rng, 12, 288) for _ in range(3)]
            if rng.random() < 0.6:
                grid[0] += grid[0] % 2  # most meshes have even rows
            cells = grid[0] * grid[1] * grid[2]
            steps = _log_int(rng, 10, 300)
            if cells <= 256 ** 3 and cells * steps <= BIGGEST:
                break
        ra = 10.0 ** rng.uniform(3.0, math.log10(min(1e6, 500.0 * grid[1] ** 2)))
        storage = rng.choice(["f32", "f32", "bf16", "f16"])
        if storage == "f32" and cells * steps > BIGGEST // 2:
            storage = "bf16"  # FP32 moves twice the bytes
        c = _cavity("", grid, rng.randint(1, 3), ra, storage, rng.choice(["two", "inplace"]), steps)
        del c["name"]
        return c
    if kind == "ensemble":
        return {"kind": kind, "count": _log_int(rng, 4, 40),
                "edges": rng.choice(["32,48,64,96", "24,40,56", "32,64", "31,45,64"]),
                "storage": rng.choice(["f32", "bf16", "f16"]), "streaming": rng.choice(["two", "inplace"]),
                "steps": _log_int(rng, 20, 100)}
    if kind == "conv":
        while True:
            n = 8 * rng.randint(1, 8)
            batch = rng.randint(1, 8)
            cin, cout = rng.choice([8, 16, 32, 64, 128]), rng.choice([16, 32, 64, 128])
            if n ** 3 * batch * cin * cout <= 64 ** 3 * 4 * 64 * 32:
                return {"kind": kind, "n": n, "batch": batch, "cin": cin, "cout": cout}
    return {"kind": kind, "net": rng.choice(["unet64", "unet64", "unet32"]), "batch": rng.randint(1, 6)}


# ---------------------------------------------------------------- inputs

def _rng(seed, salt=0):
    return np.random.default_rng([int(seed), salt])


def _modes(r, shape, count, which):
    """Sum of `count` low modes on the [z][y][x] cell centres of a box, FP32
    on the GPU, of size about one; `which`: "wall" vanishes on every wall."""
    axes = [torch.from_numpy((np.arange(n) + 0.5) / n).cuda() for n in shape]
    out = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for _ in range(count):
        a = r.uniform(-1.0, 1.0) / math.sqrt(count)
        k = r.integers(1, 4, size=3)
        f = [torch.sin(math.pi * int(k[d]) * axes[d]) if which == "wall" or d == 1
             else torch.cos(math.pi * int(k[d]) * axes[d]) for d in range(3)]
        out += a * f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    return out


def _start_fields(r, nx, ny, nz):
    """rho, u, theta of a developing convection: the conduction profile with
    smooth disturbances, a slow flow, a nearly uniform density."""
    shape = (nz, ny, nx)
    uc = MA / math.sqrt(3.0)
    y = torch.from_numpy((np.arange(ny) + 0.5) / ny).cuda()
    theta = 0.5 - y[None, :, None] + 0.2 * _modes(r, shape, 5, "side")
    u = torch.stack([0.3 * uc * _modes(r, shape, 5, "wall") for _ in range(3)])
    rho = 1.0 + 0.3 * uc * uc * _modes(r, shape, 5, "side")
    return rho.float().contiguous(), u.float().contiguous(), theta.expand(shape).float().contiguous()


def _edges(case):
    """The members' sizes, uniform over the case's edges; the same for every seed."""
    r = _rng(case["count"], 4)
    edges = [int(e) for e in case["edges"].split(",")]
    return [int(r.choice(edges)) for _ in range(case["count"])]


def _members(case, seed):
    r = _rng(seed, 1)
    return [{"grid": (e, e, e), "Ra": float(10.0 ** r.uniform(3.0, math.log10(5e5))), "wall": int(r.integers(1, 4))}
            for e in _edges(case)]


def _conv_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n, b, cin, cout = case["n"], case["batch"], case["cin"], case["cout"]
    x = torch.randn((b, n, n, n, cin), generator=g, device="cuda")
    x = torch.where(x > 0, x, 0.1 * x).to(torch.bfloat16)  # a layer's input is a layer's output
    w = torch.empty((27, cout, cin), device="cuda").uniform_(-1.0, 1.0, generator=g) * math.sqrt(6.0 / (27 * cin))
    bias = torch.empty(cout, device="cuda").uniform_(-0.1, 0.1, generator=g)
    return x, w.to(torch.bfloat16), bias


def _layers(net):
    """(cin, cout, taps) of the network's layers in parameter order."""
    _, depth, c = NETS[net]
    out = [(8, c[0], 27), (c[0], c[0], 27)]
    for l in range(1, depth + 1):
        out += [(c[l - 1], c[l], 27), (c[l], c[l], 27)]
    for l in range(depth - 1, -1, -1):
        out += [(c[l + 1], c[l], 27), (c[l], c[l], 27)]
    return out + [(c[0], 5, 1)]


def _params(net):
    """The flat FP32 parameters: those that ship with the package, or a fixed
    draw; the weights are bfloat16 numbers, as the BF16 network uses them."""
    weights = sum(a * b * t for a, b, t in _layers(net))
    biases = sum(b for _, b, _ in _layers(net))
    if net == "unet64":
        with np.load(surrogate.DEFAULT_PARAMS) as z:
            w = (z["weights_bf16"].astype(np.uint32) << 16).view(np.float32)
            b = z["biases"]
    else:
        r = _rng(7, 3)
        w = np.concatenate([r.uniform(-1, 1, a * b * t) * math.sqrt(6.0 / (t * a)) for a, b, t in _layers(net)])
        w = torch.from_numpy(w).to(torch.bfloat16).float().numpy()
        b = r.uniform(-0.1, 0.1, biases).astype(np.float32)
    assert len(w) == weights and len(b) == biases
    p, iw, ib = [], 0, 0
    for cin, cout, t in _layers(net):
        p += [w[iw:iw + cin * cout * t], b[ib:ib + cout]]
        iw, ib = iw + cin * cout * t, ib + cout
    return np.concatenate(p).astype(np.float32)


def _samples(case, seed):
    r = _rng(seed, 2)
    ra = 10.0 ** r.uniform(3.0, 6.0, case["batch"])
    wall = r.integers(1, 4, case["batch"]).astype(np.int32)
    n = NETS[case["net"]][0]
    target = None
    if case["kind"] == "gradients":
        target = torch.empty((case["batch"], n ** 3, 5), device="cuda")
        uc = MA / math.sqrt(3.0)
        for k in range(case["batch"]):
            rho, u, th = _start_fields(r, n, n, n)
            ch = [u[0] / uc, u[1] / uc, u[2] / uc, th, (rho - 1.0) / (3.0 * uc * uc)]
            target[k] = torch.stack(ch, dim=-1).reshape(n ** 3, 5)
    return ra, wall, target


# ---------------------------------------------------------------- the pass

def prepare(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        rho, u, th = _start_fields(_rng(seed), nx, ny, nz)
        torch.cuda.synchronize()
        cav = dmrt.Cavity((nx, ny, nz), case["ra"], PR, MA, case["wall"], storage=STORAGES[case["storage"]],
                          streaming=STREAMINGS[case["streaming"]], residual_interval=INTERVAL)
        dmrt.dmrt_init_fields(cav.h, rho, u, th)
        cav.sync()
        return {"kind": kind, "cav": cav, "steps": case["steps"], "rho": rho, "u": u, "theta": th}
    if kind == "ensemble":
        members = _members(case, seed)
        ens = dmrt.Ensemble(members, storage=STORAGES[case["storage"]], streaming=STREAMINGS[case["streaming"]],
                            residual_interval=INTERVAL)
        ens.autotune(trials=2)
        r = _rng(seed)
        fields = [_start_fields(r, *m["grid"]) for m in members]
        cells = [m["grid"][0] ** 3 for m in members]
        out = torch.empty(5 * sum(cells), device="cuda")  # rho, u, theta of the members, one after another
        torch.cuda.synchronize()
        views, at = [], 0
        for k, f in enumerate(fields):
            dmrt.dmrt_ensemble_init_fields(ens.e, k, *f)
            n = cells[k]
            views.append((out[at:at + n], out[at + n:at + 4 * n], out[at + 4 * n:at + 5 * n]))
            at += 5 * n
        ens.sync()
        return {"kind": kind, "ens": ens, "steps": case["steps"], "out": out, "views": views}
    if kind == "conv":
        x, w, bias = _conv_inputs(case, seed)
        y = torch.empty((*x.shape[:4], case["cout"]), dtype=torch.bfloat16, device="cuda")
        return {"kind": kind, "case": case, "x": x, "w": w, "bias": bias, "y": y}
    n, depth, channels = NETS[case["net"]]
    if case["net"] == "unet64":
        sur, _ = surrogate.load_surrogate(max_batch=case["batch"])
    else:
        sur = dmrt.Surrogate(n, depth, channels, dmrt.STORE_BF16, max_batch=case["batch"])
        sur.set_params(_params(case["net"]))
    ra, wall, target = _samples(case, seed)
    out = torch.empty((case["batch"], n ** 3, 5), device="cuda") if kind == "predict" else None
    torch.cuda.synchronize()
    return {"kind": kind, "sur": sur, "ra": ra, "wall": wall, "target": target, "out": out}


def run(state):
    kind = state["kind"]
    if kind == "cavity":
        cav = state["cav"]
        cav.step(state["steps"])
        r = cav.residual()
        nu = cav.nusselt(0)
        dmrt.dmrt_fields(cav.h, state["rho"], state["u"], state["theta"])
        return {"rho": state["rho"], "u": state["u"], "theta": state["theta"], "nu": list(nu), "residual": r}
    if kind == "ensemble":
        ens = state["ens"]
        ens.step(state["steps"])
        r = ens.residual()
        nu = ens.nusselt(0)
        for k, (rho, u, th) in enumerate(state["views"]):
            dmrt.dmrt_ensemble_fields(ens.e, k, rho, u, th)
        return {"fields": state["out"], "nu_mean": nu[:, :2].copy(), "nu_max": nu[:, 2].copy(), "residual": r}
    if kind == "conv":
        c = state["case"]
        dmrt.dmrt_nn_conv3d(state["x"], state["w"], state["bias"], state["y"], c["batch"], c["n"], c["cin"],
                            c["cout"], 3, act=1)
        return state["y"]
    if kind == "predict":
        dmrt.dmrt_surrogate_predict(state["sur"].s, state["ra"], state["wall"], state["out"])
        return state["out"]
    grad, loss = state["sur"].gradients(state["ra"], state["wall"], state["target"])
    return {"grad": grad, "loss": loss}


# ---------------------------------------------------------------- work

FLOPS_PER_CELL = 600  # FP32 operations of one coupled D3Q19 + D3Q7 collision


def _net_voxels(net):
    """(multiply-adds, of them in the first layer) of the network per sample."""
    n, depth, c = NETS[net]
    total = 8 * c[0] * 27 * n ** 3
    first = total
    total += c[0] * c[0] * 27 * n ** 3
    for l in range(1, depth + 1):
        total += (c[l - 1] + c[l]) * c[l] * 27 * (n >> l) ** 3
    for l in range(depth - 1, -1, -1):
        total += c[l + 1] * c[l] * 27 * (n >> (l + 1)) ** 3 + c[l] * c[l] * 27 * (n >> l) ** 3
    return total + c[0] * 5 * n ** 3, first


def work(case):
    kind = case["kind"]
    if kind in ("cavity", "ensemble"):
        if kind == "cavity":
            cells = case["nx"] * case["ny"] * case["nz"]
        else:
            cells = sum(e ** 3 for e in _edges(case))
        elt = 4 if case["storage"] == "f32" else 2
        # the state read and written once, the fields written once
        return {"bytes": cells * (2 * 26 * elt + 20), "flops": cells * case["steps"] * FLOPS_PER_CELL}
    if kind == "conv":
        vox = case["batch"] * case["n"] ** 3
        return {"bytes": 2 * vox * (case["cin"] + case["cout"]) + 54 * case["cin"] * case["cout"] + 4 * case["cout"],
                "flops": 2 * 27 * vox * case["cin"] * case["cout"]}
    n = NETS[case["net"]][0]
    params = sum(a * b * t + b for a, b, t in _layers(case["net"]))
    macs, first = _net_voxels(case["net"])
    io = 20 * case["batch"] * n ** 3
    if kind == "predict":
        return {"bytes": io + 2 * params, "flops": 2 * macs * case["batch"]}
    return {"bytes": io + 6 * params, "flops": 2 * (3 * macs - first) * case["batch"]}


# ---------------------------------------------------------------- 64-bit results

E19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, 1, 0),
       (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1), (-1, 0, -1), (0, 1, 1), (0, -1, 1), (0, 1, -1),
       (0, -1, -1)]
E7 = E19[:7]
CHUNK = 1 << 21  # cells collided at once


def _moment_rows():
    """The orthogonal D3Q19 moments as polynomials of the velocities."""
    rows = []
    for x, y, z in E19:
        e2 = x * x + y * y + z * z
        rows.append([1, 19 * e2 - 30, (21 * e2 * e2 - 53 * e2 + 24) / 2, x, (5 * e2 - 9) * x, y, (5 * e2 - 9) * y, z,
                     (5 * e2 - 9) * z, 3 * x * x - e2, (3 * e2 - 5) * (3 * x * x - e2), y * y - z * z,
                     (3 * e2 - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
                     (x * x - y * y) * z])
    return np.array(rows, dtype=np.float64).T


class _Box64:
    """Cavities of one shape and wall type stepped in 64 bits: state [q][member][z][y][x]."""

    def __init__(self, grid, wall, ras, fields):
        nx, ny, nz = grid
        self.grid, self.wall = grid, wall
        uc = MA / math.sqrt(3.0)
        ra = torch.tensor(ras, dtype=torch.float64, device="cuda")
        nu = uc * ny * torch.sqrt(PR / ra)
        self.gbeta = uc * uc / ny
        self.s_nu, self.q_a = 1.0 / (3.0 * nu + 0.5), 1.0 / (0.5 + 4.0 * nu / PR)
        w = [1 / 3 if not any(e) else 1 / 18 if sum(map(abs, e)) == 1 else 1 / 36 for e in E19]
        self.w = torch.tensor(w, dtype=torch.float64, device="cuda")
        self.e = torch.tensor(E19, dtype=torch.float64, device="cuda")
        M = _moment_rows()
        self.M = torch.from_numpy(M).cuda()
        self.Mi = torch.from_numpy(M.T / (M * M).sum(1)).contiguous().cuda()
        s = [1.0, 1.19, 1.4, 1.0, 1.2, 1.0, 1.2, 1.0, 1.2, 0, 1.4, 0, 1.4, 0, 0, 0, 1.98, 1.98, 1.98]
        self.s = torch.tensor(s, dtype=torch.float64, device="cuda")
        rho, th = (torch.stack([f[k] for f in fields]).double() for k in (0, 2))
        u = torch.stack([f[1] for f in fields], dim=1).double()
        m = len(fields)
        self.f = torch.empty((19, m, nz, ny, nx), dtype=torch.float64, device="cuda")
        self.g = torch.empty((7, m, nz, ny, nx), dtype=torch.float64, device="cuda")
        for i, e in enumerate(E19):
            ev = e[0] * u[0] + e[1] * u[1] + e[2] * u[2]
            self.f[i] = rho * self.w[i] * (1 + 3 * ev + 4.5 * ev * ev - 1.5 * (u * u).sum(0))
            if i < 7:
                self.g[i] = (0.25 if i == 0 else 0.125) * th * (1 + 4 * ev)
        self.member = torch.arange(m, device="cuda").repeat_interleave(nx * ny * nz)
        y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny
        self.lin = (0.5 - y)[:, None]

    @staticmethod
    def _arrive(S, e, opp, i):
        """Population i after streaming, and where its link left the box the stored opposite one."""
        out = S[opp].clone()
        dst, src = [slice(None)] * 4, [slice(None)] * 4
        for axis, d in zip((3, 2, 1), e):
            if d:
                dst[axis], src[axis] = (slice(1, None), slice(None, -1)) if d > 0 else (slice(None, -1), slice(1, None))
        out[tuple(dst)] = S[i][tuple(src)]
        return out

    def pull(self):
        f, g = torch.empty_like(self.f), torch.empty_like(self.g)
        for i, e in enumerate(E19):
            opp = E19.index((-e[0], -e[1], -e[2]))
            f[i] = self._arrive(self.f, e, opp, i)
            if i >= 7:
                continue
            g[i] = self._arrive(self.g, e, opp, i)
            for axis, d in enumerate(e):
                if d and (axis == 1 or self.wall == 2 or (self.wall == 3 and axis == 0)):
                    face = [slice(None)] * 4
                    face[3 - axis] = 0 if d > 0 else -1
                    face = tuple(face)
                    tw = d * 0.5 if axis == 1 else self.lin.squeeze(1) if axis == 0 else self.lin
                    g[i][face] = 0.25 * tw - g[i][face]
        return f, g

    def fields(self, f=None, g=None):
        if f is None:
            f, g = self.pull()
        rho = f.sum(0)
        u = torch.stack([sum(e[a] * f[i] for i, e in enumerate(E19) if e[a]) for a in range(3)]) / rho
        return rho, u, g.sum(0)

    def step(self):
        f, g = self.pull()
        cells = f[0].numel()
        F, G, f, g = self.f.view(19, cells), self.g.view(7, cells), f.view(19, cells), g.view(7, cells)
        for a in range(0, cells, CHUNK):
            b = min(cells, a + CHUNK)
            p, q, who = f[:, a:b], g[:, a:b], self.member[a:b]
            mom = self.M @ p
            rho, jx, jy, jz = mom[0], mom[3], mom[5], mom[7]
            T = q.sum(0)
            V = torch.stack([jx, jy, jz]) / rho
            jj = jx * jx + jy * jy + jz * jz
            eq = torch.zeros_like(mom)
            eq[0], eq[3], eq[5], eq[7] = rho, jx, jy, jz
            eq[1], eq[2] = -11 * rho + 19 * jj, 3 * rho - 5.5 * jj
            eq[4], eq[6], eq[8] = -2 / 3 * jx, -2 / 3 * jy, -2 / 3 * jz
            eq[9], eq[11] = 3 * jx * jx - jj, jy * jy - jz * jz
            eq[10], eq[12] = -0.5 * eq[9], -0.5 * eq[11]
            eq[13], eq[14], eq[15] = jx * jy, jy * jz, jx * jz
            eq -= mom
            nu = self.s_nu[who]
            for k in range(19):
                eq[k] *= nu if k in (9, 11, 13, 14, 15) else self.s[k]
            ev = self.e @ V
            vv = (V * V).sum(0)
            feq = rho * self.w[:, None] * (1 + 3 * ev + 4.5 * ev * ev - 1.5 * vv)
            force = 3.0 * self.gbeta * T * (self.e[:, 2:3] - V[2]) * feq
            F[:, a:b] = p + self.Mi @ eq + force
            # energy: moments T; fluxes; 6 g0 - sum; 3 (x pair) - pairs; y pair - z pair
            px, py, pz = q[1] + q[2], q[3] + q[4], q[5] + q[6]
            qa = self.q_a[who]
            d = [qa * (V[k] * T - (q[2 * k + 1] - q[2 * k + 2])) / 2 for k in range(3)]
            d4 = (0.75 * T - (6 * q[0] - px - py - pz)) / 42
            d5, d6 = -(2 * px - py - pz) / 12, -(py - pz) / 4
            G[0, a:b] = q[0] + 6 * d4
            for k, even in enumerate((2 * d5 - d4, -d4 - d5 + d6, -d4 - d5 - d6)):
                G[2 * k + 1, a:b] = q[2 * k + 1] + even + d[k]
                G[2 * k + 2, a:b] = q[2 * k + 2] + even - d[k]

    def advance(self, steps):
        """Steps, then the residual of each member from the last two points."""
        points, r = [], torch.full((self.f.shape[1],), math.inf, dtype=torch.float64)
        for s in range(steps):
            if (s + 1) % INTERVAL == 0:
                _, u, th = self.fields()
                points.append((u.movedim(1, 0).flatten(1), th.flatten(1)))
                if len(points) > 2:
                    points.pop(0)
            self.step()
        if len(points) == 2:
            rel = [((b - a).norm(dim=1) / b.norm(dim=1)) for a, b in zip(*points)]
            r = (torch.maximum(*rel) / INTERVAL).cpu()
        return r.numpy()

    def nusselt(self, th):
        """Nu_3D, Nu_2D, Nu_max on the hot wall of each member, from theta [member][z][y][x]."""
        nx, ny, _ = self.grid
        local = -ny * (-4.0 + 9.0 * th[:, :, 0] - th[:, :, 1]) / 3.0
        mid = local[:, :, (nx - 1) // 2:nx // 2 + 1]
        return torch.stack([local.mean((1, 2)), mid.mean((1, 2)), local.amax((1, 2))], dim=1).cpu().numpy()


def _unpack(net, p):
    out, at = [], 0
    for cin, cout, t in _layers(net):
        out.append((p[at:at + t * cout * cin].view(t, cout, cin), p[at + t * cout * cin:at + t * cout * cin + cout]))
        at += t * cout * cin + cout
    return out


def _conv64(x, w, bias, act):
    """Channels-last convolution, zero outside: x [b][z][y][x][cin], w [taps][cout][cin]."""
    n = x.shape[1]
    if w.shape[0] == 1:
        return x @ w[0].T + bias
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    y = bias.expand(*x.shape[:4], w.shape[1])
    for t in range(27):
        z0, y0, x0 = t // 9, t // 3 % 3, t % 3
        y = y + xp[:, z0:z0 + n, y0:y0 + n, x0:x0 + n] @ w[t].T
    return torch.where(y > 0, y, 0.1 * y) if act else y


def _net64(net, p, ra, wall):
    n, depth, _ = NETS[net]
    b = len(ra)
    c = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n
    x = torch.zeros((b, n, n, n, 8), dtype=torch.float64, device="cuda")
    for k in range(b):
        x[k, ..., 0] = (math.log10(ra[k]) - 4.5) / 1.5
        x[k, ..., int(wall[k])] = 1.0
    x[..., 4] = 2 * c - 1
    x[..., 5] = (2 * c - 1)[:, None]
    x[..., 6] = (2 * c - 1)[:, None, None]
    x[..., 7] = (0.5 - c)[:, None]
    P = iter(_unpack(net, p))
    skip = []
    for level in range(depth + 1):
        if level:
            m = x.shape[1] // 2
            x = x.reshape(b, m, 2, m, 2, m, 2, -1).mean(dim=(2, 4, 6))
        for _ in range(2):
            x = _conv64(x, *next(P), True)
        skip.append(x)
    for level in range(depth - 1, -1, -1):
        x = _conv64(x, *next(P), True)
        for d in (1, 2, 3):
            x = x.repeat_interleave(2, dim=d)
        x = _conv64(x + skip[level], *next(P), True)
    return _conv64(x, *next(P), False).reshape(b, n ** 3, 5)


def exact(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        grid = (case["nx"], case["ny"], case["nz"])
        rho, u, th = _start_fields(_rng(seed), *grid)
        box = _Box64(grid, case["wall"], [case["ra"]], [(rho, u, th)])
        r = box.advance(case["steps"])
        rho, u, th = box.fields()
        nu = [float(v) for v in box.nusselt(th)[0]]
        if case["storage"] != "f32":
            nu[2] = None  # the largest of single cells: with 16-bit storage, of their stochastic rounding
        return {"rho": rho[0], "u": u[:, 0], "theta": th[0], "nu": nu, "residual": float(r[0])}
    if kind == "ensemble":
        members = _members(case, seed)
        gen = _rng(seed)
        starts = [_start_fields(gen, *m["grid"]) for m in members]
        fields = [None] * len(members)
        nu, res = np.zeros((len(members), 3)), np.zeros(len(members))
        for key in sorted({(m["grid"], m["wall"]) for m in members}):
            at = [k for k, m in enumerate(members) if (m["grid"], m["wall"]) == key]
            box = _Box64(key[0], key[1], [members[k]["Ra"] for k in at], [starts[k] for k in at])
            r = box.advance(case["steps"])
            rho, u, th = box.fields()
            v = box.nusselt(th)
            for j, k in enumerate(at):
                nu[k], res[k] = v[j], r[j]
                fields[k] = torch.cat([rho[j].flatten(), u[:, j].flatten(), th[j].flatten()])
            del box, rho, u, th
        return {"fields": torch.cat(fields), "nu_mean": nu[:, :2].copy(),
                "nu_max": nu[:, 2].copy() if case["storage"] == "f32" else None, "residual": res}
    if kind == "conv":
        x, w, bias = _conv_inputs(case, seed)
        return _conv64(x.double(), w.double(), bias.double(), True)
    ra, wall, target = _samples(case, seed)
    p = torch.from_numpy(_params(case["net"])).double().cuda()
    if kind == "predict":
        with torch.no_grad():
            return _net64(case["net"], p, ra, wall)
    p.requires_grad_(True)
    loss = ((_net64(case["net"], p, ra, wall) - target.double()) ** 2).mean()
    loss.backward()
    return {"grad": p.grad.cpu().numpy(), "loss": float(loss.detach())}
