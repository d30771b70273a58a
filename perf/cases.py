"""The work that programs using this package have it do, as cases to measure.

Every case is a job a user's program runs through the public entry points of
``paper_2602_05017_gb300`` on data it already holds on the GPU: the initial field goes in
(``set_density``), the steps run, the field is read where it lies (the ``field_tensor`` view).  Grids,
substrate parameters, agents and initial fields follow the workloads of ``inputs.py``.

``exact`` restates the method in plain torch at 64 bits: per axis and substrate the dense
inverse of the Appendix A matrix applied as a matrix product, so it shares neither code nor
operation order with the kernels.
"""
import math

import numpy as np
import torch

from paper_2602_05017_gb300 import autotune, inputs
from paper_2602_05017_gb300.adjoint import lod_steps
from paper_2602_05017_gb300.binding import BioFVM, BioFVMBatch

DX, DT, TARGET = 20.0, 0.01, 38.0
# substrate parameters of the 400^3 x 4 workload, repeated for more substrates
D_ALL = (1e5, 1e3, 5e2, 1e2, 2e4, 3e3, 8e4, 2e2)
LAM_ALL = (0.1, 0.01, 0.4, 1e-3, 0.05, 0.2, 1.0, 0.002)
ELEM = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}


def _step(name, precision, nx, ny, nz, ns, steps, agents, dirichlet=False, nodes=0,
          field="uniform"):
    return dict(name=name, kind="step", precision=precision, nx=nx, ny=ny, nz=nz, ns=ns,
                steps=steps, agents=agents, dirichlet=dirichlet, nodes=nodes, field=field)


def listed():
    return [
        # one call per time step on a small tissue sample, as an agent-based program that
        # interleaves its own cell updates makes it: latency and launches
        _step("call_fp32_41x37x29_s2", "fp32", 41, 37, 29, 2, 1, 60, dirichlet=True),
        # the smallest workload of the benchmark: FP64, 200 cells, 100 steps a call
        _step("sample_fp64_50c_s1", "fp64", 50, 50, 50, 1, 100, 200),
        # the headline workload: 400^3 x 4 with a million agents, FP64 and FP32
        _step("tissue_fp64_400c_s4", "fp64", 400, 400, 400, 4, 8, 1_000_000),
        _step("tissue_fp32_400c_s4", "fp32", 400, 400, 400, 4, 8, 1_000_000),
        # the large Dirichlet workload's line lengths (1200), blobs as the initial field
        _step("organ_fp32_1200x400x900_s2", "fp32", 1200, 400, 900, 2, 2, 1_000_000,
              dirichlet=True, field="blobs"),
        # the 5 mm cube of the end-to-end run, FP64, cells that stay where they are
        _step("cube_fp64_250c_s1", "fp64", 250, 250, 250, 1, 20, 1000, field="gauss"),
        # the same cube in FP32 with cells that move every step: source lists rebuilt on the
        # device before each one-step call
        dict(name="moving_fp32_250c_s1", kind="moving", precision="fp32", nx=250, ny=250, nz=250,
             ns=1, steps=10, agents=1000),
        # half-precision storage on a mid-sized field
        _step("half_fp16_320x256x288_s4", "fp16", 320, 256, 288, 4, 8, 100_000),
        # the batched configuration's recipe (edges 32..192, 1..8 substrates, FP32)
        dict(name="batch_fp32_48env", kind="batch", envs=48, lo=32, hi=192, smax=8, steps=8),
        # many small samples advanced together (parameter studies): edges 16..64
        dict(name="batch_fp32_small_60env", kind="batch", envs=60, lo=16, hi=64, smax=4,
             steps=40),
        # parameter fitting through the differentiable run: the adjoint workload's grid, and an
        # uneven one in FP32
        dict(name="adjoint_fp64_128c_s2", kind="adjoint", precision="fp64", nx=128, ny=128,
             nz=128, ns=2, steps=20, every=10),
        dict(name="adjoint_fp32_113x97x121_s3", kind="adjoint", precision="fp32", nx=113, ny=97,
             nz=121, ns=3, steps=20, every=10),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "moving", "batch", "adjoint", "adjoint"])
    if kind == "batch":
        hi = _log_int(rng, 24, 192)
        lo = rng.randint(max(8, hi // 6), hi - 4)
        smax = rng.randint(1, 8)
        envs = max(1, min(_log_int(rng, 2, 60), int(6e8 / (hi ** 3 * (smax + 1)))))
        return dict(kind="batch", envs=envs, lo=lo, hi=hi, smax=smax, steps=_log_int(rng, 1, 40))
    if kind == "adjoint":
        nx, ny, nz = (_log_int(rng, 12, 128) for _ in range(3))
        return dict(kind="adjoint", precision=rng.choice(["fp64", "fp32"]), nx=nx, ny=ny, nz=nz,
                    ns=rng.randint(1, 3), steps=rng.randint(3, 20), every=rng.randint(2, 10))
    precision = rng.choice(["fp64", "fp64", "fp32", "fp32", "fp32", "bf16", "fp16"])
    if kind == "moving" and precision not in ("fp64", "fp32"):
        precision = "fp32"
    cells = math.exp(rng.uniform(math.log(5e3), math.log(1e8)))  # voxel-substrates in all
    ns = rng.choice([1, 1, 2, 2, 3, 4, 4, 5, 6, 8])
    a, b = math.exp(rng.uniform(-0.7, 0.7)), math.exp(rng.uniform(-0.7, 0.7))
    edge = (cells / ns) ** (1.0 / 3.0)
    nx, ny, nz = (max(4, min(900, int(round(edge * f)))) for f in (a, b, 1.0 / (a * b)))
    if precision in ("bf16", "fp16"):  # 16-bit rows are multiples of 8 elements
        nx = max(8, min(400, nx // 8 * 8))
        ny, nz = min(400, ny), min(400, nz)
    agents = _log_int(rng, 1, max(1, min(1_000_000, nx * ny * nz // 50)))
    cost = 1.1e9 / (nx * ny * nz * ns)  # steps that keep a draw below the largest listed case
    steps = max(1, min(_log_int(rng, 1, 100), int(cost)))
    if kind == "moving":
        return dict(kind="moving", precision=precision, nx=nx, ny=ny, nz=nz, ns=ns,
                    steps=min(steps, 20), agents=agents)
    nodes = 0
    if precision in ("fp64", "fp32") and rng.random() < 0.15:
        nodes = _log_int(rng, 1, max(1, nx * ny * nz // 200))
    case = _step("", precision, nx, ny, nz, ns, steps, agents, rng.random() < 0.4, nodes,
                 rng.choice(["uniform", "blobs", "gauss"]))
    del case["name"]
    return case


# -- inputs --------------------------------------------------------------------------------
def _params(ns):
    k = [s % len(D_ALL) for s in range(ns)]
    return np.array([D_ALL[i] for i in k]), np.array([LAM_ALL[i] for i in k])


def _field(case, seed, dtype):
    """Initial field [nz, ny, nx, ns] on the GPU: uniform in [0, 38], a sum of Gaussian blobs, or
    one Gaussian in the middle."""
    nz, ny, nx, ns = case["nz"], case["ny"], case["nx"], case["ns"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case.get("field", "uniform") == "uniform":
        r = torch.rand((nz, ny, nx, ns), generator=g, device="cuda",
                       dtype=torch.float64 if dtype == torch.float64 else torch.float32)
        return r.mul_(TARGET).to(dtype)
    rng = np.random.default_rng(seed)
    n = 8 if case["field"] == "blobs" else 1
    out = torch.zeros((nz, ny, nx, ns), device="cuda", dtype=dtype)
    for _ in range(n):
        fac = []
        for m in (nz, ny, nx):
            c = rng.uniform(0.2, 0.8) if n > 1 else 0.5
            sig = rng.uniform(0.08, 0.25) if n > 1 else 0.2
            x = (np.arange(m) + 0.5) / m
            fac.append(np.exp(-0.5 * ((x - c) / sig) ** 2))
        amp = rng.uniform(1.0, TARGET, ns)
        z, y, xs = (torch.as_tensor(f, device="cuda", dtype=dtype) for f in fac)
        xs = xs[:, None] * torch.as_tensor(amp, device="cuda", dtype=dtype)
        out.addcmul_((z[:, None] * y[None, :])[:, :, None, None], xs[None, None])
    return out


def _agents(case, seed, n=None):
    rng = np.random.default_rng(seed + 1)
    return inputs.random_agents(rng, case["nx"] * case["ny"] * case["nz"], case["ns"],
                                case["agents"] if n is None else n)


def _dirichlet(case):
    if not case.get("dirichlet"):
        return None, None
    ns = case["ns"]
    on = np.array([1 if s % 2 == 0 else 0 for s in range(ns)], dtype=np.uint8)
    return on, np.where(on == 1, TARGET, 0.0)


def _nodes(case, seed):
    rng = np.random.default_rng(seed + 2)
    return inputs.random_nodes(rng, case["nx"] * case["ny"] * case["nz"], case["ns"],
                               case["nodes"])


def _moves(case, seed):
    """Voxel of every agent before each step: a walk of one voxel along a random axis a step."""
    g = torch.Generator(device="cuda").manual_seed(seed + 3)
    n, size = case["agents"], torch.tensor([case["nx"], case["ny"], case["nz"]], device="cuda")
    pos = (torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64) * size).long()
    pos = torch.minimum(pos, size - 1)
    out = []
    for _ in range(case["steps"]):
        axis = torch.randint(0, 3, (n, 1), generator=g, device="cuda")
        way = torch.randint(0, 2, (n, 1), generator=g, device="cuda") * 2 - 1
        pos = pos.scatter_add(1, axis, way).clamp(min=0).minimum(size - 1)
        out.append(((pos[:, 2] * case["ny"] + pos[:, 1]) * case["nx"] + pos[:, 0]).contiguous())
    return out


def _envs(case, seed):
    rng = np.random.default_rng(1000 + case["lo"] + 7 * case["hi"])  # the study's grids
    grids = [(int(rng.integers(case["lo"], case["hi"] + 1)), int(rng.integers(1, case["smax"] + 1)))
             for _ in range(case["envs"])]
    rng = np.random.default_rng(seed)
    envs = []
    for e, (n, s) in enumerate(grids):
        w = inputs.Workload(f"env{e}", n, n, n, s, DX, DT,
                            np.exp(rng.uniform(math.log(1e2), math.log(1e5), s)),
                            np.exp(rng.uniform(math.log(1e-3), 0.0, s)), case["steps"])
        w.voxel, w.secretion, w.target, w.uptake = inputs.random_agents(
            rng, n ** 3, s, max(1, n ** 3 // 64))
        envs.append(w)
    return envs


def _adjoint_inputs(case, seed):
    nx, ny, nz, ns = case["nx"], case["ny"], case["nz"], case["ns"]
    rng = np.random.default_rng(seed)
    nvox = nx * ny * nz
    na = max(1, nvox // 100)
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    agents = dict(voxel=rng.choice(nvox, size=na, replace=False).astype(np.int64),
                  target=np.full((na, ns), TARGET), weight=None)
    D, lam = _params(ns)
    n_probe = min(4096, nvox * ns)
    up = lambda a: torch.as_tensor(a, device="cuda")
    return dict(rho0=_field(case, seed, dtype), agents=agents,
                secretion=up(np.exp(rng.uniform(math.log(1e-3), math.log(10.0), (na, ns)))),
                uptake=up(rng.uniform(0.0, 1.0, (na, ns))), D=up(D), lam=up(lam),
                probe=up(rng.choice(nvox * ns, size=n_probe, replace=False)),
                want=up(rng.uniform(0.0, TARGET, n_probe)).to(dtype))


# -- one pass ------------------------------------------------------------------------------
def _view(sim, owner):
    """The field where it lies, for the program to read: a view that keeps the simulation that
    owns the memory alive."""
    t = sim.field_tensor()
    t.owner = owner
    return t


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        envs = _envs(case, seed)
        tiles = autotune.tile_shapes(envs, autotune.load(autotune.default_cache_path()))
        sim = BioFVMBatch(envs, precision="fp32", tile_m=tiles)
        rho = []
        for e, (w, b) in enumerate(zip(envs, sim.envs)):
            b.set_sources(w.voxel, w.secretion, w.target, w.uptake)
            rho.append(_field(dict(nx=w.nx, ny=w.ny, nz=w.nz, ns=w.ns), seed + e, torch.float32))
        return dict(case=case, sim=sim, rho=rho, field=[_view(b, sim) for b in sim.envs])
    nx, ny, nz, ns, precision = (case[k] for k in ("nx", "ny", "nz", "ns", "precision"))
    D, lam = _params(ns)
    on, val = _dirichlet(case)
    sim = BioFVM(nx, ny, nz, ns, DX, DT, D, lam, on, val, precision=precision)
    if kind == "adjoint":
        st = _adjoint_inputs(case, seed)
        for k in ("rho0", "secretion", "uptake", "D", "lam"):
            st[k].requires_grad_(True)
        return dict(case=case, sim=sim, **st)
    rho = _field(case, seed, sim._field_dtype())
    if kind == "moving":
        _, sec, tgt, upt = _agents(case, seed)
        sim.reserve_agents(case["agents"])
        up = lambda a: torch.as_tensor(a, device="cuda")
        return dict(case=case, sim=sim, rho=rho, moves=_moves(case, seed), sec=up(sec),
                    tgt=up(tgt), upt=up(upt), field=_view(sim, sim))
    if case["nodes"]:
        sim.set_dirichlet_nodes(*_nodes(case, seed))
    sim.set_sources(*_agents(case, seed))
    return dict(case=case, sim=sim, rho=rho, field=_view(sim, sim))


def run(st):
    case, sim = st["case"], st["sim"]
    kind = case["kind"]
    if kind == "step":
        sim.set_density(st["rho"])
        sim.step(case["steps"])
        return st["field"]
    if kind == "moving":
        sim.set_density(st["rho"])
        for voxel in st["moves"]:
            sim.set_sources_device(voxel, st["sec"], st["tgt"], st["upt"])
            sim.step(1)
        return st["field"]
    if kind == "batch":
        for env, rho in zip(sim.envs, st["rho"]):
            env.set_density(rho)
        sim.step(case["steps"])
        return st["field"]
    wrt = [st[k] for k in ("rho0", "secretion", "uptake", "D", "lam")]
    out = lod_steps(st["rho0"], st["secretion"], st["D"], st["lam"], sim, st["agents"],
                    case["steps"], case["every"], uptake=st["uptake"])
    loss = (out.reshape(-1)[st["probe"]] - st["want"]).square().sum()
    grads = torch.autograd.grad(loss, wrt)
    return [out.detach(), *grads]


def work(case):
    """Inputs read once and outputs written once; Eq. 2's five operations per element of a
    Thomas line, three sweeps a step."""
    if case["kind"] == "batch":
        nel = sum(w.nx * w.ny * w.nz * w.ns for w in _envs(case, 0))
        return {"bytes": 8.0 * nel, "flops": 15.0 * nel * case["steps"]}
    nel = float(case["nx"]) * case["ny"] * case["nz"] * case["ns"]
    esz = ELEM[case["precision"]]
    if case["kind"] == "adjoint":
        # forward, then per step the reverse sweeps and the two sums per sweep behind dD and
        # dlambda (six operations); the field in, the result, its gradient out
        na = max(1, case["nx"] * case["ny"] * case["nz"] // 100) * case["ns"]
        return {"bytes": 3.0 * esz * nel + 6 * 8.0 * na,
                "flops": nel * case["steps"] * (15.0 + 15.0 + 18.0)}
    per_step = 8.0 * case["agents"] * (1 + 3 * case["ns"])
    return {"bytes": 2.0 * esz * nel + per_step * (case["steps"] if case["kind"] == "moving" else 1),
            "flops": 15.0 * nel * case["steps"]}


def tolerance(case):
    precision = case.get("precision", "fp32")
    if case["kind"] == "adjoint":
        # the sums behind dD nearly cancel: FP32 states leave about 1e-5 of them
        return {"rel": 3e-12, "max": 1e-10} if precision == "fp64" else {"rel": 2e-5, "max": 1e-3}
    # about four times the distance from exact() over the ranges of draw()
    return {"fp64": {"rel": 2e-13, "max": 2e-12}, "fp32": {"rel": 2e-6, "max": 2e-5},
            "fp16": {"rel": 5e-3, "max": 5e-2}, "bf16": {"rel": 2e-2, "max": 3e-1}}[precision]


# -- the same at 64 bits -------------------------------------------------------------------
def _inverse(n, D, lam):
    """[ns, n, n] inverses of (1 + lam dt/3) I + (D dt/dx^2) L, L the zero-flux second
    difference of an axis of n voxels."""
    L = torch.zeros((n, n), dtype=torch.float64, device=D.device)
    i = torch.arange(n - 1, device=D.device)
    L[i, i] += 1.0
    L[i + 1, i + 1] += 1.0
    L[i, i + 1] -= 1.0
    L[i + 1, i] -= 1.0
    eye = torch.eye(n, dtype=torch.float64, device=D.device)
    A = (1.0 + lam * (DT / 3.0))[:, None, None] * eye + (D * (DT / DX ** 2))[:, None, None] * L
    return torch.linalg.inv(A)


def _source_terms(shape, voxel, sec, tgt, upt):
    """alpha and 1 / (1 + beta) of every element, [nz, ny, nx, ns] -> [ns, nz, ny, nx]."""
    nz, ny, nx, ns = shape
    a = torch.zeros((nz * ny * nx, ns), dtype=torch.float64, device="cuda")
    b = torch.zeros_like(a)
    a = a.index_add(0, voxel, DT * sec * tgt)
    b = b.index_add(0, voxel, DT * (sec + upt))
    turn = lambda t: t.reshape(nz, ny, nx, ns).permute(3, 0, 1, 2).contiguous()
    return turn(a), 1.0 / (1.0 + turn(b))


def _exact_steps(rho, inv, src, steps, on=None, val=None, nodes=None):
    """``steps`` steps of u [ns, nz, ny, nx]; src(k) gives (alpha, scale) of step k."""
    u = rho.double().permute(3, 0, 1, 2).contiguous()
    S, nz, ny, nx = u.shape

    def bc(v):
        if on is None and nodes is None:
            return v
        for s in range(S):
            if on is not None and on[s]:
                w = v[s]
                for face in (w[0], w[-1], w[:, 0], w[:, -1], w[:, :, 0], w[:, :, -1]):
                    face.fill_(float(val[s]))
        if nodes is not None:
            vox, sub, value = nodes
            v.view(S, -1)[sub, vox] = value
        return v
    for k in range(steps):
        alpha, scale = src(k)
        u = bc((u + alpha) * scale)
        u = bc(torch.matmul(u.reshape(S, nz * ny, nx), inv[0]).reshape(S, nz, ny, nx))
        u = bc(torch.matmul(inv[1][:, None], u))
        u = bc(torch.matmul(inv[2], u.reshape(S, nz, ny * nx)).reshape(S, nz, ny, nx))
    return u.permute(1, 2, 3, 0)


def _last_nodes(case, seed):
    """The node list with the last value of a repeated (voxel, substrate)."""
    if not case.get("nodes"):
        return None
    keep = {(int(v), int(s)): float(x) for v, s, x in zip(*_nodes(case, seed))}
    up = lambda a, t: torch.tensor(a, device="cuda", dtype=t)
    return (up([k[0] for k in keep], torch.int64), up([k[1] for k in keep], torch.int64),
            up(list(keep.values()), torch.float64))


def exact(case, seed):
    up = lambda a: torch.as_tensor(a, device="cuda", dtype=torch.float64)
    if case["kind"] == "batch":
        out = []
        for e, w in enumerate(_envs(case, seed)):
            rho = _field(dict(nx=w.nx, ny=w.ny, nz=w.nz, ns=w.ns), seed + e, torch.float32)
            inv = [_inverse(w.nx, up(w.D), up(w.lam))] * 3
            terms = _source_terms(w.shape, torch.as_tensor(w.voxel, device="cuda"),
                                  up(w.secretion), up(w.target), up(w.uptake))
            out.append(_exact_steps(rho, inv, lambda k: terms, case["steps"]).contiguous())
        return out
    nx, ny, nz, ns = (case[k] for k in ("nx", "ny", "nz", "ns"))
    shape = (nz, ny, nx, ns)
    D, lam = (up(a) for a in _params(ns))
    if case["kind"] == "adjoint":
        st = _adjoint_inputs(case, seed)
        wrt = [st["rho0"].double(), st["secretion"], st["uptake"], st["D"], st["lam"]]
        for t in wrt:
            t.requires_grad_(True)
        rho0, sec, upt, D, lam = wrt
        inv = [_inverse(n, D, lam) for n in (nx, ny, nz)]
        terms = _source_terms(shape, torch.as_tensor(st["agents"]["voxel"], device="cuda"), sec,
                              up(st["agents"]["target"]), upt)
        out = _exact_steps(rho0, inv, lambda k: terms, case["steps"]).contiguous()
        loss = (out.reshape(-1)[st["probe"]] - st["want"].double()).square().sum()
        return [out.detach(), *torch.autograd.grad(loss, wrt)]
    dtype = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16,
             "bf16": torch.bfloat16}[case["precision"]]
    inv = [_inverse(n, D, lam) for n in (nx, ny, nz)]
    rho = _field(case, seed, dtype)
    voxel, sec, tgt, upt = _agents(case, seed)
    sec, tgt, upt = up(sec), up(tgt), up(upt)
    if case["kind"] == "moving":
        moves = _moves(case, seed)
        src = lambda k: _source_terms(shape, moves[k], sec, tgt, upt)
    else:
        terms = _source_terms(shape, torch.as_tensor(voxel, device="cuda"), sec, tgt, upt)
        src = lambda k: terms
    on, val = _dirichlet(case)
    return _exact_steps(rho, inv, src, case["steps"], on, val, _last_nodes(case, seed)).contiguous()
