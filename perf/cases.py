"""What the library is timed on: passes through its public entry points.

A case is one of these kinds of use:

  step      advance one periodic box: ``lbp_step``, then the fields, the
            populations, the particles and (where kept) the VACF and MSD are
            read into device buffers;
  pinned    the drag experiment: a particle held in a uniform stream with a
            body force that holds the mean flow;
  ensemble  many boxes of different size and viscosity in one handle, one
            particle each, with the VACF kept per particle;
  exchange  a host controller that hands over forces and takes back positions
            and velocities every step (``lbp_step_exchange``, page-locked);
  train     one gradient of a velocity-relaxation loss through
            ``adjoint.trajectory``: the run is set up, recorded and swept back;
  adjoint   record and reverse sweep on a handle that is kept;
  correlate the VACF of a trajectory the caller holds
            (``lbp_vacf_correlate_noalloc``).

``exact`` computes the same in FP64 with plain torch (D3Q15 BGK with the
Stokeslet-fit coupling, arXiv:1909.13412, Eqs. 1-20); gradients by autograd.
"""
import math

import numpy as np
import torch

from paper_1909_13412_gb300 import adjoint, lbp

STORAGE = {"f32": lbp.LBP_F32, "bf16": lbp.LBP_BF16, "f16": lbp.LBP_F16}
MODE = {"stokeslet": lbp.LBP_STOKESLET, "pointwise": lbp.LBP_POINTWISE, "brownian": lbp.LBP_BROWNIAN}
ENSEMBLE_TAUS = (0.6, 0.8, 1.0)


def listed():
    box = {"tau": 0.8, "mode": "stokeslet", "mass": 10.0, "gamma": 0.5}
    brownian = dict(box, kind="step", kT=1e-4)
    return [
        # the single-particle relaxation run (configs/config1): a small box, all latency
        dict(box, name="relax_32_f32", kind="step", nx=32, ny=32, nz=32, storage="f32", particles=1, kT=0.0,
             vacf_lag=-1, steps=100),
        # the drag experiment in the paper's own box (100^3, tau of its Fig. 1), 20 steps between feedbacks
        dict(box, name="drag_100_f32", kind="pinned", nx=100, ny=100, nz=100, storage="f32", tau=0.5534,
             particles=1, kT=0.0, radius=0.4, steps=20),
        # a small Brownian suspension with its VACF and MSD (the fluctuation-dissipation experiment)
        dict(brownian, name="brownian_64_f32", nx=64, ny=64, nz=64, storage="f32", particles=256, vacf_lag=200,
             steps=128),
        # the Brownian suspension at its stated size (configs/config2), VACF and MSD to lag 5000
        dict(brownian, name="brownian_128_f32", nx=128, ny=128, nz=128, storage="f32", particles=2000,
             vacf_lag=5000, steps=128),
        # the throughput workload (configs/config3): 1 GB of populations a buffer
        dict(brownian, name="brownian_256_f32", nx=256, ny=256, nz=256, storage="f32", particles=16384,
             vacf_lag=5000, steps=64),
        # the same with 2-byte storage
        dict(brownian, name="brownian_256_bf16", nx=256, ny=256, nz=256, storage="bf16", particles=16384,
             vacf_lag=5000, steps=64),
        # an odd, elongated channel-like box in half precision with point-wise friction (Eq. 7)
        dict(brownian, name="channel_odd_f16", nx=333, ny=75, nz=91, storage="f16", mode="pointwise",
             particles=2048, vacf_lag=-1, steps=64),
        # the replica ensemble (configs/config4): 48 x 64^3 + 16 x 96^3 + 4 x 160^3, per-particle VACF
        dict(box, name="ensemble_68_f32", kind="ensemble", n64=48, n96=16, n160=4, n_odd=0, storage="f32",
             kT=1e-4, vacf_lag=5000, steps=32),
        # a host controller in the loop of the throughput workload
        dict(box, name="exchange_256_f32", kind="exchange", nx=256, ny=256, nz=256, storage="f32",
             particles=16384, kT=1e-4, steps=16),
        # one training step of the differentiable run (configs/config5), through torch.autograd
        dict(box, name="train_64_f32", kind="train", nx=64, ny=64, nz=64, storage="f32", particles=8, kT=0.0,
             steps=200, every=50),
        # gradients of the suspension at the throughput size, on a kept handle
        dict(box, name="adjoint_256_f32", kind="adjoint", nx=256, ny=256, nz=256, storage="f32",
             particles=16384, kT=1e-4, steps=20, every=10),
        # the VACF of a recorded trajectory: 512 particles over 4096 samples
        dict(name="correlate_4096", kind="correlate", samples=4096, components=1536, vacf_lag=1000),
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sizes(most):
        # the nodes of the box over the logarithm of the range, in unequal edges
        n = log_uniform(32 ** 3, most)
        a, b = math.exp(rng.uniform(-0.4, 0.4)), math.exp(rng.uniform(-0.4, 0.4))
        edge = n ** (1.0 / 3.0)
        step = rng.choice((1, 1, 4, 32))
        nx = max(24, int(edge * a) // step * step)
        ny = max(16, int(edge * b))
        return {"nx": nx, "ny": ny, "nz": max(8, int(n / (nx * ny)))}

    def nodes(s):
        return s["nx"] * s["ny"] * s["nz"]

    kind = rng.choice(("step", "step", "step", "pinned", "ensemble", "exchange", "train", "adjoint", "correlate"))
    tau = round(rng.uniform(0.6, 1.2), 3)
    common = {"kind": kind, "tau": tau, "mass": round(rng.uniform(5.0, 20.0), 2),
              "gamma": round(min(0.5, 6.0 * math.pi * (tau - 0.5) / 3.0 * 0.6) * rng.uniform(0.5, 1.0), 3),
              "mode": "stokeslet"}
    if kind == "correlate":
        return {"kind": kind, "samples": log_uniform(100, 4096), "components": log_uniform(3, 1536),
                "vacf_lag": log_uniform(10, 1000)}
    storage = rng.choice(("f32", "f32", "bf16", "f16"))
    if kind == "ensemble":
        return dict(common, n64=rng.randint(1, 32), n96=rng.randint(0, 8), n160=rng.randint(0, 2),
                    n_odd=rng.randint(0, 8), storage=storage, kT=1e-4, vacf_lag=log_uniform(100, 5000),
                    steps=rng.randint(8, 32))
    if kind == "pinned":
        s = sizes(128 ** 3)
        return dict(common, **s, storage="f32", particles=1, kT=0.0, radius=round(rng.uniform(0.2, 0.6), 2),
                    steps=20)
    most = {"step": 250 ** 3, "exchange": 250 ** 3, "train": 64 ** 3, "adjoint": 160 ** 3}[kind]
    s = sizes(most)
    # from a handful of particles up to twice the density of the throughput workload
    np_ = max(1, min(16384, log_uniform(1, max(2, nodes(s) // 512))))
    c = dict(common, **s, storage=storage, particles=np_, kT=rng.choice((0.0, 1e-4, 1e-4)))
    if kind == "step":
        c.update(mode=rng.choice(("stokeslet", "stokeslet", "pointwise", "brownian")),
                 vacf_lag=rng.choice((-1, log_uniform(20, 5000))), steps=rng.randint(16, 64))
    elif kind == "exchange":
        c.update(steps=rng.randint(2, 16))
    else:
        c.update(storage="f32", steps=rng.randint(10, 40 if kind == "adjoint" else 100), every=rng.randint(3, 20))
        c["particles"] = min(np_, 2000)
    return c


# ------------------------------------------------------------------ inputs
def boxes_of(case):
    """[(nx, ny, nz, tau)] of the case's handle."""
    if case["kind"] != "ensemble":
        return [(case["nx"], case["ny"], case["nz"], case["tau"])]
    boxes = []
    for count, edge in ((case["n64"], 64), (case["n96"], 96), (case["n160"], 160)):
        boxes += [(edge, edge, edge, ENSEMBLE_TAUS[i % 3]) for i in range(count)]
    boxes += [(41 + 7 * i, 50, 37, ENSEMBLE_TAUS[i % 3]) for i in range(case["n_odd"])]
    return boxes


def flow_of(shape, rng, amplitude=1e-3):
    """A smooth divergence-free flow [3, nz, ny, nx]: three shear modes, u_k independent of x_k."""
    nx, ny, nz = shape
    axes = [torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n) for n in (nx, ny, nz)]
    x, y, z = axes[0][None, None, :], axes[1][None, :, None], axes[2][:, None, None]
    u = torch.empty((3, nz, ny, nx), dtype=torch.float64, device="cuda")
    for k, (p, q) in enumerate(((y, z), (z, x), (x, y))):
        f = rng.uniform(0.0, 2.0 * math.pi, 2)
        u[k] = amplitude * torch.sin(p + f[0]) * torch.cos(2.0 * q + f[1])
    return u


def inputs_of(case, seed):
    """The run's inputs by box: particles (r, v, mass, gamma, radius as numpy) and the flow."""
    rng = np.random.default_rng([seed, 1909])
    out = []
    for nx, ny, nz, tau in boxes_of(case):
        n = 1 if case["kind"] == "ensemble" else case["particles"]
        edge = np.array([nx, ny, nz], dtype=np.float64)
        gamma = min(case["gamma"], 6.0 * math.pi * (tau - 0.5) / 3.0 * 1.2)
        radius = gamma / (6.0 * math.pi * (tau - 0.5) / 3.0)
        r = np.minimum(rng.random((n, 3)) * edge, np.nextafter(edge, 0.0))
        v = rng.standard_normal((n, 3)) * math.sqrt(max(case["kT"], 1e-5) / case["mass"])
        flow = None
        if case["kind"] == "pinned":
            # held at a cell centre of a uniform stream along x
            r = np.floor(r) + 0.5
            v = np.zeros((n, 3))
            radius = case["radius"]
            gamma = 6.0 * math.pi * (tau - 0.5) / 3.0 * radius
            flow = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device="cuda")
            flow[0] = 1e-4 * rng.uniform(0.5, 1.5)
        elif case["kT"] == 0.0:
            # kicked particles in a fluid at rest, near cell centres
            r = np.floor(r) + rng.uniform(0.35, 0.65, (n, 3))
            v *= 0.01 / np.linalg.norm(v, axis=1, keepdims=True)
        else:
            flow = flow_of((nx, ny, nz), rng)
        out.append({"tau": tau, "shape": (nx, ny, nz), "flow": flow, "r": r, "v": v,
                    "mass": np.full(n, case["mass"]), "gamma": np.full(n, gamma), "radius": np.full(n, radius)})
    return out


def forces_of(case, seed):
    """A controller's forces, one set per step."""
    rng = np.random.default_rng([seed, 20])
    return rng.standard_normal((case["steps"], case["particles"], 3)) * 1e-3


def loss_gradients(case, seed):
    """dL/dV and dL/dr of some loss on the trajectory, for the reverse sweep on a kept handle."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["steps"], case["particles"], 3)
    return [torch.randn(shape, dtype=torch.float64, device="cuda", generator=g) * s for s in (1.0, 1e-2)]


def trajectory_of(case, seed):
    """A trajectory of Ornstein-Uhlenbeck-like velocities [samples, components], FP32."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    white = torch.randn((case["samples"] + 32, case["components"]), device="cuda", generator=g)
    kernel = torch.exp(-torch.arange(32, device="cuda", dtype=torch.float32) / 8.0)
    out = torch.zeros((case["samples"], case["components"]), device="cuda")
    for k in range(32):
        out += kernel[k] * white[32 - k:32 - k + case["samples"]]
    return (out * 3e-3).contiguous()


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def empty(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device="cuda")


def make_handle(case, seed):
    boxes, ins = boxes_of(case), inputs_of(case, seed)
    if case["kind"] == "ensemble":
        h = lbp.lbp_create_batch(boxes, precision=STORAGE[case["storage"]])
    else:
        h = lbp.lbp_create(*boxes[0], precision=STORAGE[case["storage"]])
    flows = [b["flow"] for b in ins]
    if flows[0] is not None:
        lbp.lbp_set_fluid(h, None, torch.cat([f.reshape(3, -1) for f in flows], 1).contiguous())
    for k, b in enumerate(ins):
        lbp.lbp_particles_add_to(h, k, b["r"], b["v"], b["mass"], b["gamma"], b["radius"])
    lbp.lbp_particles_set_params(h, kT=case["kT"], seed=seed, mode=MODE[case["mode"]])
    return h, ins


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "correlate":
        s["samples"] = trajectory_of(case, seed)
        s["csum"] = empty(case["vacf_lag"] + 1)
        s["counts"] = empty(case["vacf_lag"] + 1, dtype=torch.int64)
        return s
    if kind == "train":
        b = inputs_of(case, seed)[0]
        s["spec"] = adjoint.RunSpec(*b["shape"], steps=case["steps"], checkpoint_every=case["every"], kT_seed=seed)
        s["fixed"] = {"f0": None if b["flow"] is None else equilibrium(b["flow"]) + weights().reshape(-1, 1, 1, 1)}
        s["params"] = [torch.tensor(b["tau"], dtype=torch.float64, device="cuda")] + [
            cuda(b[k]) for k in ("gamma", "radius", "mass", "v", "r")]
        for p in s["params"]:
            p.requires_grad_(True)
        return s
    h, ins = make_handle(case, seed)
    n = sum(len(b["mass"]) for b in ins)
    s["h"] = h
    s["r"], s["v"], s["f_h"], s["f_r"] = (empty(n, 3) for _ in range(4))
    if kind == "adjoint":
        s["g_v"], s["g_r"] = loss_gradients(case, seed)
        s["v_traj"], s["r_traj"] = empty(case["steps"], n, 3), empty(case["steps"], n, 3)
        s["grads"] = {"tau": empty(1), "kT": empty(1), "gamma": empty(n), "radius": empty(n), "mass": empty(n),
                      "v0": empty(n, 3), "r0": empty(n, 3), "f0": empty(15, h.N)}
        return s
    if kind == "exchange":
        s["forces"] = torch.from_numpy(forces_of(case, seed))
        s["f_ext"], s["r_host"], s["v_host"] = (torch.zeros((n, 3), dtype=torch.float64).pin_memory()
                                                for _ in range(3))
    s["u"] = empty(3, h.N)
    s["f"] = empty(15, h.N)
    if kind == "pinned":
        lbp.lbp_particles_set_external_force(h, None, np.ones(n, np.uint8))
        lbp.lbp_set_body_force(h, (3e-9, 0.0, 0.0))
    if case.get("vacf_lag", -1) >= 0:
        k1 = case["vacf_lag"] + 1
        if kind == "ensemble":
            lbp.lbp_vacf_configure_ex(h, case["vacf_lag"], True)
            s["csum"] = empty(n, k1)
        else:
            lbp.lbp_vacf_configure(h, case["vacf_lag"])
            s["csum"], s["msum"] = empty(k1), empty(k1)
        s["counts"] = empty(k1, dtype=torch.int64)
    return s


# -------------------------------------------------------------------- run
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "correlate":
        lbp.lbp_vacf_correlate_noalloc(s["samples"], case["samples"], case["components"], case["vacf_lag"],
                                       case["components"] // 3, s["csum"], s["counts"])
        return {"csum": s["csum"], "counts": s["counts"]}
    if kind == "train":
        tau, gamma, radius, mass, v0, r0 = s["params"]
        v_traj, r_traj = adjoint.trajectory(tau, gamma, radius, mass, v0, r0, s["spec"], kT=case["kT"], **s["fixed"])
        loss = adjoint.relaxation_loss(v_traj, v0.detach(), 20.0)
        grads = torch.autograd.grad(loss, s["params"])
        return {"loss": loss.detach(), "v": v_traj.detach(), "r": r_traj.detach(), "grads": grads}
    h = s["h"]
    if kind == "adjoint":
        lbp.lbp_adjoint_record(h, case["steps"], case["every"], s["v_traj"], s["r_traj"])
        lbp.lbp_adjoint_backward(h, case["steps"], s["g_v"], s["g_r"], s["grads"])
        return {"v": s["v_traj"], "r": s["r_traj"], "grads": s["grads"]}
    if kind == "exchange":
        for f in s["forces"]:
            s["f_ext"].copy_(f)
            lbp.lbp_step_exchange(h, s["f_ext"], s["r_host"], s["v_host"])
    else:
        lbp.lbp_step(h, case["steps"])
    lbp.lbp_read_fields(h, None, s["u"])
    lbp.lbp_read_populations(h, s["f"])
    out = {"u": s["u"], "f": s["f"]}
    if kind == "exchange":
        out.update(r=s["r_host"], v=s["v_host"])
        return out
    lbp.lbp_particles_read(h, s["r"], s["v"], s["f_h"], s["f_r"])
    out.update({k: s[k] for k in ("r", "v", "f_h", "f_r")})
    if "msum" in s:
        lbp.lbp_vacf_read(h, s["csum"], s["counts"])
        lbp.lbp_msd_read(h, s["msum"], s["counts"])
        out.update({k: s[k] for k in ("csum", "msum", "counts")})
    elif "csum" in s:
        lbp.lbp_vacf_read_per_particle(h, s["csum"], s["counts"])
        out.update({k: s[k] for k in ("csum", "counts")})
    return out


def work(case):
    """Bytes and operations of a pass: every step reads and writes the
    populations (15 each per node, in the storage type), an adjoint step reads
    two sets and writes one; what is read out is written once as FP64."""
    kind = case["kind"]
    if kind == "correlate":
        t, c, k = case["samples"], case["components"], case["vacf_lag"] + 1
        return {"bytes": 4 * t * c + 16 * k, "flops": 2 * c * sum(max(0, t - i) for i in range(k))}
    n = sum(nx * ny * nz for nx, ny, nz, _ in boxes_of(case))
    size = 4 if case["storage"] == "f32" else 2
    steps = case["steps"]
    particles = len(boxes_of(case)) if kind == "ensemble" else case["particles"]
    step = n * 30 * size + particles * 8 * 14 * size
    flops = n * 190 * steps
    if kind in ("train", "adjoint"):
        # record, one replayed segment state less than its length, reverse steps
        replay = steps - -(-steps // case["every"])
        total = step * (steps + replay) + (n * 45 * 4 + particles * 8 * 28 * 4) * steps
        return {"bytes": total + (n * 15 * 12 if kind == "adjoint" else 0), "flops": 4 * flops}
    # the flow and the populations read out: both read every population, and write 3 and 15 FP64 values
    return {"bytes": step * steps + n * (2 * 15 * size + 18 * 8), "flops": flops}


# ------------------------------------------------------- the same in 64 bits
VELOCITIES = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 1), (-1, -1, -1),
              (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1))


def velocities():
    return torch.tensor(VELOCITIES, dtype=torch.float64, device="cuda")


def weights():
    return torch.tensor([2.0 / 9.0] + [1.0 / 9.0] * 6 + [1.0 / 72.0] * 8, dtype=torch.float64, device="cuda")


def equilibrium(u, drho=None):
    """f^eq - w (Eq. 17) of the flow u [3, ...]."""
    shape = u.shape[1:]
    u = u.reshape(3, -1)
    eu = velocities() @ u
    g = 4.5 * eu * eu + 3.0 * eu - 1.5 * (u * u).sum(0)
    if drho is not None:
        g = g + drho.reshape(-1)
    return (weights()[:, None] * g).reshape(15, *shape)


def high64(a, b):
    """The high 64 bits of the unsigned products a b (int64 tensors holding uint64 bits)."""
    mask = 0xFFFFFFFF
    a0, a1, b0, b1 = a & mask, (a >> 32) & mask, b & mask, (b >> 32) & mask
    low, m1, m2 = a0 * b0, a1 * b0, a0 * b1
    mid = ((low >> 32) & mask) + (m1 & mask) + (m2 & mask)
    return a1 * b1 + ((m1 >> 32) & mask) + ((m2 >> 32) & mask) + (mid >> 32)


def signed(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def noise(step, first, n, seed):
    """xi [n, 3] of a step: Philox-4x64-10 (Salmon et al., SC'11), counter (step, particle), key (seed, 0)."""
    zero = torch.zeros(n, dtype=torch.int64, device="cuda")
    c = [zero + step, torch.arange(first, first + n, device="cuda"), zero, zero]
    m0, m1 = (zero + signed(m) for m in (0xD2E7470EE14C6C93, 0xCA5A826395121157))
    for k in range(10):
        k0, k1 = signed(seed + k * 0x9E3779B97F4A7C15), signed(k * 0xBB67AE8584CAA73B)
        c = [high64(m1, c[2]) ^ c[1] ^ k0, m1 * c[2], high64(m0, c[0]) ^ c[3] ^ k1, m0 * c[0]]
    bits = torch.stack(c[:3], 1)
    k53 = (bits >> 11) & ((1 << 53) - 1)
    return math.sqrt(3.0) * ((k53.double() + 0.5) * 2.0 ** -52 - 1.0)


def step64(g, r, v, omega, p, xi, f_ext=None):
    """One time step in deviation form: (g, r, v) -> (g, r, v, F_H, F_R); p holds the run's constants."""
    e, w = velocities(), weights()
    nz, ny, nx = g.shape[1:]
    g = torch.stack([torch.roll(g[a], (c[2], c[1], c[0]), (0, 1, 2)) if a else g[0]
                     for a, c in enumerate(VELOCITIES)]).reshape(15, -1)
    u = e.T @ g
    edge = torch.tensor([nx, ny, nz], dtype=torch.float64, device="cuda")
    base = torch.floor(r.detach())
    q = r - base
    corner = torch.tensor([(c & 1, c >> 1 & 1, c >> 2) for c in range(8)], dtype=torch.float64, device="cuda")
    node = torch.remainder(base[:, None] + corner, edge).long()
    node = ((node[..., 2] * ny + node[..., 1]) * nx + node[..., 0]).reshape(-1)
    weight = torch.where(corner > 0, q[:, None], 1.0 - q[:, None]).prod(2)
    up = u[:, node].T.reshape(-1, 8, 3)
    gamma, radius = p["gamma"][:, None], p["radius"][:, None]
    if p["mode"] == "stokeslet":
        rel = up - v[:, None]
        mean = rel.mean(1)
        size = mean.norm(dim=1, keepdim=True)
        moving = size > 0
        en = torch.where(moving, mean / torch.where(moving, size, torch.ones_like(size)), torch.zeros_like(mean))
        d = corner - q[:, None]
        rp = d.norm(dim=2)
        away = 1.0 / rp
        k1 = 1.0 - 0.75 * radius * away
        k2 = 0.75 * radius * (d * en[:, None]).sum(2) * away ** 3
        a = k1[..., None] * en[:, None] - k2[..., None] * d
        den = (a * a).sum((1, 2))
        f_h = gamma * ((rel * a).sum((1, 2)) / torch.where(den > 0, den, torch.ones_like(den)))[:, None] * en
    elif p["mode"] == "pointwise":
        f_h = -gamma * (v - (weight[..., None] * up).sum(1))
    else:
        f_h = -gamma * v
    force = torch.zeros_like(u) + p["body"][:, None]
    if p["mode"] != "brownian":
        share = -(weight[..., None] * f_h[:, None]).reshape(-1, 3)
        force = force.index_add(1, node, share.T)
    f_r = torch.sqrt(2.0 * gamma * p["kT"]) * xi if p["kT"] > 0 else torch.zeros_like(v)
    if not p["pinned"]:
        push = f_h + f_r if f_ext is None else f_h + f_r + f_ext
        v = v + push / p["mass"][:, None]
        r = torch.remainder(r + v, edge)
    eu = e @ u
    geq = w[:, None] * (g.sum(0) + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0))
    g = g + omega * (geq - g) + 3.0 * w[:, None] * (e @ force)
    return g.reshape(15, nz, ny, nx), r, v, f_h, f_r


def constants(case, b):
    body = (3e-9, 0.0, 0.0) if case["kind"] == "pinned" else (0.0, 0.0, 0.0)
    return {"mode": case["mode"], "kT": case["kT"], "pinned": case["kind"] == "pinned",
            "body": torch.tensor(body, dtype=torch.float64, device="cuda"),
            **{k: cuda(b[k]) for k in ("gamma", "radius", "mass")}}


def start64(b):
    nx, ny, nz = b["shape"]
    g = torch.zeros((15, nz, ny, nx), dtype=torch.float64, device="cuda") if b["flow"] is None \
        else equilibrium(b["flow"])
    return g, cuda(b["r"]), cuda(b["v"])


def gradients64(case, seed):
    """The trajectory and the gradients of a recorded run, by autograd over checkpointed steps."""
    from torch.utils.checkpoint import checkpoint
    b = inputs_of(case, seed)[0]
    p = constants(case, b)
    tau = torch.tensor(b["tau"], dtype=torch.float64, device="cuda", requires_grad=True)
    kT = torch.tensor(float(case["kT"]), dtype=torch.float64, device="cuda", requires_grad=case["kT"] > 0)
    p["kT"] = kT
    g, r, v = start64(b)
    leaves = {"tau": tau, "kT": kT, "gamma": p["gamma"], "radius": p["radius"], "mass": p["mass"], "v0": v, "r0": r,
              "f0": g}
    for x in (p["gamma"], p["radius"], p["mass"], g, r, v):
        x.requires_grad_(True)
    vs, rs = [], []
    for n in range(case["steps"]):
        xi = noise(n, 0, r.shape[0], seed)
        g, r, v = checkpoint(lambda g, r, v, xi: step64(g, r, v, 1.0 / tau, p, xi)[:3], g, r, v, xi,
                             use_reentrant=False)
        vs.append(v)
        rs.append(r)
    v_traj, r_traj = torch.stack(vs), torch.stack(rs)
    if case["kind"] == "train":
        t = torch.arange(1, case["steps"] + 1, dtype=torch.float64, device="cuda")
        target = leaves["v0"].detach() * torch.exp(-t / 20.0)[:, None, None]
        loss = ((v_traj - target) ** 2).mean()
        names = ("tau", "gamma", "radius", "mass", "v0", "r0")
        return {"loss": loss.detach(), "v": v_traj.detach(), "r": r_traj.detach(),
                "grads": torch.autograd.grad(loss, [leaves[k] for k in names])}
    g_v, g_r = loss_gradients(case, seed)
    names = [k for k in leaves if k != "kT" or case["kT"] > 0]
    got = dict(zip(names, torch.autograd.grad((v_traj * g_v).sum() + (r_traj * g_r).sum(), [leaves[k] for k in names])))
    out = {k: None for k in leaves}
    out.update(got)
    out["tau"] = out["tau"].reshape(1)
    out["kT"] = out["kT"].reshape(1) if out["kT"] is not None else None
    out["f0"] = out["f0"].reshape(15, -1)
    return {"v": v_traj.detach(), "r": r_traj.detach(), "grads": out}


def exact(case, seed):
    kind = case["kind"]
    if kind == "correlate":
        x, t, k1 = trajectory_of(case, seed).double(), case["samples"], case["vacf_lag"] + 1
        power = torch.fft.rfft(x, n=t + k1, dim=0).abs().square().sum(1)
        csum = torch.fft.irfft(power, n=t + k1)[:k1]
        csum[min(t, k1):] = 0.0
        return {"csum": csum, "counts": None}
    if kind in ("train", "adjoint"):
        # every step's state is kept: a few hundred steps of a small box, none of a large one
        nodes = case["nx"] * case["ny"] * case["nz"]
        return gradients64(case, seed) if nodes * case["steps"] <= 64 ** 3 * 250 else None
    out = {k: [] for k in ("u", "f", "r", "v", "f_h", "f_r")}
    samples = []
    first = 0
    forces = cuda(forces_of(case, seed)) if kind == "exchange" else None
    for b in inputs_of(case, seed):
        p = constants(case, b)
        g, r, v = start64(b)
        kept = []
        for n in range(case["steps"]):
            xi = noise(n, first, r.shape[0], seed)
            g, r, v, f_h, f_r = step64(g, r, v, 1.0 / b["tau"], p, xi, None if forces is None else forces[n])
            kept.append(v)
        first += r.shape[0]
        samples.append(torch.stack(kept))
        streamed = torch.stack([torch.roll(g[a], (c[2], c[1], c[0]), (0, 1, 2))
                                for a, c in enumerate(VELOCITIES)]).reshape(15, -1)
        out["u"].append(velocities().T @ streamed)
        out["f"].append((g + weights().reshape(-1, 1, 1, 1)).reshape(15, -1))
        for k, x in (("r", r), ("v", v), ("f_h", f_h), ("f_r", f_r)):
            out[k].append(x)
        del g, streamed
    out = {k: torch.cat(x, 1 if k in ("u", "f") else 0) for k, x in out.items()}
    if kind == "exchange":
        return {"u": out["u"], "f": out["f"], "r": out["r"].cpu(), "v": out["v"].cpu()}
    if case["kT"] == 0.0:
        out["f_r"] = None
    if case.get("vacf_lag", -1) >= 0:
        # all lags of the pass's few samples; later lags have no pairs yet
        t, k1 = case["steps"], case["vacf_lag"] + 1
        vel = torch.cat(samples, 1)
        pos = vel.cumsum(0)
        rows = 1 if kind == "step" else vel.shape[1]
        csum = torch.zeros((rows, k1), dtype=torch.float64, device="cuda")
        msum = torch.zeros(k1, dtype=torch.float64, device="cuda")
        for k in range(min(t, k1)):
            c = (vel[:t - k] * vel[k:]).sum((0, 2))
            csum[:, k] = c.sum() if kind == "step" else c
            msum[k] = (pos[k:] - pos[:t - k]).square().sum()
        out["counts"] = None
        out["csum"] = csum[0] if kind == "step" else csum
        if kind == "step":
            out["msum"] = msum
    return out
