"""The performance cases of the stepper: what a user's program has it do.

Four kinds of call, each through a public entry point of the package:

  step     `Simulation.step(n)` on one 2D or 3D grid in FP64, FP32 or FP16
           storage, launched pass by pass or replayed as a CUDA graph
  monitor  the same followed by `Simulation.observe()`: a run that watches its
           energy and phase volume every n steps
  batch    `Batch.step(n)` on many independent 2D grids of uneven sizes
  forward  `ac_net_forward`: one learned jump of a batch of fields
  train    `ac_net_loss_grads` and `ac_net_adam`: one training step of the jump
           network

Sizes, interface widths and initial states follow the repository's workloads
(`paper_2105_09671_gb300.workloads`): h = 1 / nx, dt = 0.1 h^2, eps a few
cells, a random state of amplitude 0.1 or a tanh circle / sphere.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2105_09671_gb300 as ac
from paper_2105_09671_gb300 import _lib as lib

TORCH = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16}
ITEM = {"f64": 8, "f32": 4, "f16s": 2}
CHANNELS = 32      # of the jump network's hidden layers
JUMP = 16          # Euler steps that one learned jump stands for
BATCH_SIZES = tuple(range(64, 1025, 32))


def _step(name, shape, dtype, n, init, eps_cells, graph, kind="step"):
    nz, ny, nx = (0,) * (3 - len(shape)) + tuple(shape)
    return dict(name=name, kind=kind, nz=nz, ny=ny, nx=nx, dtype=dtype, n=n, init=init, eps_cells=eps_cells,
                graph=graph)


def listed():
    return [
        # The radius-law experiment: a 64^2 circle in FP64, replayed as a
        # graph.  The smallest call, bound by the latency of a step.
        _step("circle_64_f64", (64, 64), "f64", 100, "sphere", 0.96, True),
        # A 2D run of the size of the paper's tables, issued launch by launch
        # as a first program does.
        _step("table_200x400_f32", (200, 400), "f32", 100, "sphere", 2.4, False),
        # A mid-sized separation run that reads its energy every 100 steps.
        _step("monitor_1024_f32", (1024, 1024), "f32", 100, "random", 4.0, True, kind="monitor"),
        # The large 2D separation run, in FP32 and in FP64.
        _step("separation_4096_f32", (4096, 4096), "f32", 60, "random", 16.384, True),
        _step("separation_4096_f64", (4096, 4096), "f64", 10, "random", 16.384, True),
        # 3D runs of the size of the paper's tables: a sphere on 100^3 (no
        # axis a multiple of a tile), and FP64 on 200 x 100 x 100.
        _step("sphere_100_f32", (100, 100, 100), "f32", 100, "sphere", 2.9, False),
        _step("box_200x100x100_f64", (100, 100, 200), "f64", 50, "sphere", 2.9, False),
        # FP16 storage on 256^3, and the 512^3 throughput run.
        _step("sphere_256_f16s", (256, 256, 256), "f16s", 40, "sphere", 0.77, True),
        _step("sphere_512_f32", (512, 512, 512), "f32", 20, "sphere", 1.54, True),
        # A parameter study: many uneven grids advanced together.
        dict(name="batch_64", kind="batch", count=64, smallest=64, largest=1024, dtype="f32", n=200),
        # One learned jump of the 1024^2 evaluation field, and one training
        # step on a pool of 256^2 trajectories.
        dict(name="forward_1024", kind="forward", ndim=2, batch=1, nz=1, ny=1024, nx=1024),
        dict(name="train_256_pool32", kind="train", ndim=2, batch=32, nz=1, ny=256, nx=256),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["step"] * 5 + ["monitor", "batch", "forward", "train"])
    if kind == "batch":
        smallest = rng.choice(BATCH_SIZES[:8])
        return dict(kind=kind, count=rng.randint(8, 64), smallest=smallest,
                    largest=rng.choice([s for s in BATCH_SIZES if s > smallest and s <= 1024]),
                    dtype=rng.choice(["f32", "f32", "f16s"]), n=rng.randint(20, 200))
    if kind in ("forward", "train"):
        ndim = rng.choice([2, 2, 3])
        if ndim == 2:
            nz, ny, nx = 1, _log(rng, 48, 1024), _log(rng, 48, 1024)
        else:
            nz, ny, nx = (_log(rng, 16, 64) for _ in range(3))
        # the pool stays within the listed case's 32 x 256^2 pixels of work
        room = (1 << 21) // (nz * ny * nx * (3 if ndim == 3 else 1))
        return dict(kind=kind, ndim=ndim, batch=max(1, min(_log(rng, 1, 32), room)), nz=nz, ny=ny, nx=nx)
    ndim = rng.choice([2, 3])
    dtype = rng.choice(["f64", "f32", "f32", "f16s"])
    if ndim == 2:
        shape = (_log(rng, 24, 4096), _log(rng, 24, 4096))
    else:
        shape = tuple(_log(rng, 12, 512) for _ in range(3))
    cells = math.prod(shape)
    # no more work than the largest listed case of the storage type
    most = max(4, int((1.6e8 if dtype == "f64" else 2.5e9) / cells))
    c = _step("", shape, dtype, min(rng.randint(10, 120), most), rng.choice(["sphere", "random"]),
              round(rng.uniform(1.5, 6.0), 3), rng.random() < 0.5, kind=kind)
    del c["name"]
    return c


# ------------------------------------------------------------- the inputs --

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _shape(c):
    return (c["ny"], c["nx"]) if not c["nz"] or c.get("ndim") == 2 else (c["nz"], c["ny"], c["nx"])


def _initial(shape, init, eps, h, seed):
    """A random state of amplitude 0.1, or a tanh circle / sphere whose place
    and radius the seed draws, on cells of size h; FP64 on the GPU."""
    g = _gen(seed)
    if init == "random":
        return 0.1 * (2.0 * torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") - 1.0)
    place = torch.rand(4, generator=g, dtype=torch.float64, device="cuda").tolist()
    span = h * min(shape)
    r2 = 0.0
    for axis, n in enumerate(shape):
        x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h
        x = x - (0.5 + 0.1 * (place[axis] - 0.5)) * n * h
        r2 = r2 + (x * x).reshape([-1 if a == axis else 1 for a in range(len(shape))])
    return torch.tanh(((0.2 + 0.1 * place[3]) * span - r2.sqrt()) / (math.sqrt(2.0) * eps))


def _grid(c):
    h = 1.0 / c["nx"]
    return h, c["eps_cells"] * h, 0.1 * h * h


def _batch_specs(c, seed):
    """(shape, h, eps, dt, initial state) of every grid.  The sizes are the
    study's own, the same for every seed."""
    sizes = random.Random(c["count"] * 4096 + c["largest"])
    rng = random.Random(seed)
    out = []
    for i in range(c["count"]):
        n = sizes.choice([s for s in BATCH_SIZES if c["smallest"] <= s <= c["largest"]])
        h = 1.0 / n
        eps = rng.uniform(3.0, 6.0) * h
        out.append(((n, n), h, eps, 0.1 * h * h, "sphere" if i % 2 == 0 else "random"))
    return out


def _parameters(ndim, seed):
    """[(W, b)] of the six layers in FP32: He-normal weights, small biases, and
    a last layer of the size that training gives it.  W is [taps, in, out]."""
    g = _gen(seed + 7)
    taps = 3 ** ndim
    out = []
    for layer in range(6):
        cin, cout = (1 if layer == 0 else CHANNELS), (1 if layer == 5 else CHANNELS)
        sd = 0.05 if layer == 5 else math.sqrt(2.0 / (taps * cin))
        w = sd * torch.randn((taps, cin, cout), generator=g, dtype=torch.float64, device="cuda")
        b = 0.02 * torch.randn((cout,), generator=g, dtype=torch.float64, device="cuda")
        out.append((w.float(), b.float()))
    return out


def _net_fields(c, seed):
    """FP32 inputs of the network: random and tanh states, as a pool holds."""
    shape = _shape(c)
    h = 1.0 / c["nx"]
    return torch.stack([_initial(shape, "random" if i % 2 == 0 else "sphere", 4.0 * h, h, seed * 64 + i)
                        for i in range(c["batch"])]).float().contiguous()


def _targets(phi, c):
    """Plausible targets of a jump: the reaction alone, over the jump's time."""
    return (phi + JUMP * (0.1 / 16.0) * (phi - phi ** 3)).contiguous()


SCALE = JUMP * 0.1 / 16.0  # n dt / eps^2 at eps = 4 h


class _Stream:
    """The one stream of the program, on which all its calls are ordered (a
    graph replay needs another than the default stream)."""
    kept = None

    @classmethod
    def get(cls):
        if cls.kept is None:
            cls.kept = torch.cuda.Stream()
        return cls.kept


def prepare(case, seed):
    c = case
    if c["kind"] in ("step", "monitor"):
        shape = _shape(c)
        h, eps, dt = _grid(c)
        sim = ac.Simulation(shape, h, eps, dt, dtype=c["dtype"], stream=_Stream.get())
        sim.phi.copy_(_initial(shape, c["init"], eps, h, seed))
        sim.set_graph(c["graph"])
        torch.cuda.synchronize()
        return dict(case=c, sim=sim)
    if c["kind"] == "batch":
        specs = _batch_specs(c, seed)
        batch = ac.Batch([s[:4] for s in specs], dtype=c["dtype"], stream=_Stream.get())
        for i, (shape, h, eps, _, init) in enumerate(specs):
            batch.phi(i).copy_(_initial(shape, init, eps, h, seed * 64 + i))
        torch.cuda.synchronize()
        return dict(case=c, batch=batch)
    net = _Net(c["ndim"], seed)
    phi = _net_fields(c, seed)
    state = dict(case=c, net=net, phi=phi)
    if c["kind"] == "forward":
        state["out"] = torch.empty_like(phi)
    else:
        state["target"] = _targets(phi, c)
    torch.cuda.synchronize()
    return state


class _Net:
    """A network handle that its program destroys when done with it."""

    def __init__(self, ndim, seed):
        self.handle = lib.ac_net_create(ndim, torch.cuda.current_stream().cuda_stream)
        flat = torch.cat([torch.cat([w.reshape(-1), b]) for w, b in _parameters(ndim, seed)])
        lib.ac_net_set_params(self.handle, flat.cpu().numpy())

    def __del__(self):
        lib.ac_net_destroy(self.handle)


def run(state):
    c = state["case"]
    if c["kind"] == "step":
        state["sim"].step(c["n"])
        return state["sim"].phi
    if c["kind"] == "monitor":
        state["sim"].step(c["n"])
        energy, volume, _ = state["sim"].observe()
        return dict(phi=state["sim"].phi, observed=np.array([energy, volume]))
    if c["kind"] == "batch":
        state["batch"].step(c["n"])
        return [state["batch"].phi(i) for i in range(c["count"])]
    phi = state["phi"]
    if c["kind"] == "forward":
        lib.ac_net_forward(state["net"].handle, phi.data_ptr(), state["out"].data_ptr(), c["batch"], c["nx"], c["ny"],
                           c["nz"], SCALE)
        return state["out"]
    loss, grads = lib.ac_net_loss_grads(state["net"].handle, phi.data_ptr(), state["target"].data_ptr(), c["batch"],
                                        c["nx"], c["ny"], c["nz"], SCALE, want_grads=True)
    lib.ac_net_adam(state["net"].handle, 1e-3)
    return dict(loss=loss, grads=grads)


# ------------------------------------------------ what a pass can't do without --

def work(case):
    c = case
    if c["kind"] in ("step", "monitor"):
        shape = _shape(c)
        cells = math.prod(shape)
        per = 12 if len(shape) == 2 else 14  # operations of one update
        return {"bytes": 2 * ITEM[c["dtype"]] * cells, "flops": per * cells * c["n"]}
    if c["kind"] == "batch":
        cells = sum(s[0][0] * s[0][1] for s in _batch_specs(c, 0))
        return {"bytes": 2 * ITEM[c["dtype"]] * cells, "flops": 12 * cells * c["n"]}
    cells = c["batch"] * c["nz"] * c["ny"] * c["nx"]
    macs = 3 ** c["ndim"] * (4 * CHANNELS * CHANNELS + 2 * CHANNELS)
    # forward; a training step adds the data and the weight gradients
    return {"bytes": 8 * cells, "flops": 2 * macs * cells * (3 if c["kind"] == "train" else 1)}


def tolerance(case):
    """About four times the largest error against `exact` seen over the ranges."""
    c = case
    if c["kind"] == "forward":   # BF16 activations; seen up to 2.8e-4
        return {"rel": 1.2e-3, "max": 4e-2}
    if c["kind"] == "train":     # gradients through five BF16 layers; seen up to 1.7e-2
        return {"rel": 3e-2, "max": 3e-1}
    # seen up to 3.1e-16, 2.7e-7 and 4.1e-4 (one rounding to FP16 per pass)
    return {"f64": {"rel": 1.3e-15, "max": 2e-14}, "f32": {"rel": 1.2e-6, "max": 2e-5},
            "f16s": {"rel": 1.7e-3, "max": 2e-2}}[c["dtype"]]


# --------------------------------------------------- the same in 64 bits --

def _advance(phi, h, eps, dt, n):
    """n explicit Euler steps with replicated boundary cells, FP64."""
    dims = range(phi.dim())
    for _ in range(n):
        lap = phi * (-2.0 * phi.dim())
        for d in dims:
            m = phi.shape[d]
            lo, hi = phi.narrow(d, 0, 1), phi.narrow(d, m - 1, 1)
            lap += torch.cat([lo, phi.narrow(d, 0, m - 1)], d)
            lap += torch.cat([phi.narrow(d, 1, m - 1), hi], d)
        phi = phi + dt * ((phi - phi * phi * phi) / eps ** 2 + lap / h ** 2)
    return phi


def _energy(phi, h, eps):
    e = ((phi * phi - 1.0) ** 2).sum().item() / 4.0 / eps ** 2
    for d in range(phi.dim()):
        e += 0.5 * (phi.diff(dim=d) ** 2).sum().item() / h ** 2
    return h ** phi.dim() * e, h ** phi.dim() * (1.0 + phi).sum().item() / 2.0


def _gelu(x):
    return 0.5 * x * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (x + 0.044715 * x ** 3)))


def _conv(x, w, b, ndim):
    """Replicate-padded cross-correlation; x is [batch, *space, in]."""
    for d in range(1, ndim + 1):
        m = x.shape[d]
        x = torch.cat([x.narrow(d, 0, 1), x, x.narrow(d, m - 1, 1)], d)
    out = b
    for t in range(3 ** ndim):
        y, r = x, t
        for d in range(ndim, 0, -1):  # the last axis (x) is fastest in t
            y = y.narrow(d, r % 3, x.shape[d] - 2)
            r //= 3
        out = out + y @ w[t]
    return out


def _network(phi, params, ndim):
    x = phi.unsqueeze(-1)
    for layer, (w, b) in enumerate(params):
        x = _conv(x, w, b, ndim)
        if layer < 5:
            x = _gelu(x)
    return phi + SCALE * x.squeeze(-1)


def exact(case, seed):
    c = case
    if c["kind"] in ("step", "monitor"):
        h, eps, dt = _grid(c)
        phi = _advance(_initial(_shape(c), c["init"], eps, h, seed).to(TORCH[c["dtype"]]).double(), h, eps, dt, c["n"])
        if c["kind"] == "step":
            return phi
        return dict(phi=phi, observed=np.array(_energy(phi, h, eps)))
    if c["kind"] == "batch":
        return [_advance(_initial(shape, init, eps, h, seed * 64 + i).to(TORCH[c["dtype"]]).double(), h, eps, dt, c["n"])
                for i, (shape, h, eps, dt, init) in enumerate(_batch_specs(c, seed))]
    phi32 = _net_fields(c, seed)
    params = [(w.double(), b.double()) for w, b in _parameters(c["ndim"], seed)]
    phi = phi32.double()
    if c["kind"] == "forward":
        with torch.no_grad():
            return _network(phi, params, c["ndim"])
    target = _targets(phi32, c).double()
    leaves = [t.requires_grad_() for pair in params for t in pair]
    total = 0.0
    for i in range(c["batch"]):  # one field at a time: its graph is freed before the next
        loss = (((_network(phi[i:i + 1], params, c["ndim"]) - target[i:i + 1]) / SCALE) ** 2).sum() / phi.numel()
        loss.backward()
        total += loss.item()
    return dict(loss=total, grads=torch.cat([t.grad.reshape(-1) for t in leaves]).cpu().numpy())
