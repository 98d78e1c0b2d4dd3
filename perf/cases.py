"""The performance cases of this framework: what its users have it do, and what each call returns.

Each family goes through the entry points of ``paper_2311_18126_gb300``:

* ``step``     one or more implicit steps of a batch of clamped rods from a given state: state, frames and
               natural curvatures in, the new state and frames out (what a controller or a rollout does).
* ``robots``   the same for limbed star robots crawling on the ground (joints, ground contact, friction).
* ``coil``     the same for one helical rod whose turns lie on each other (edge-edge contact).
* ``grippers`` the same for grippers of several fingers that touch each other (contact groups, friction).
* ``adjoint``  the step's adjoint: gradients of a loss on the new state.
* ``rollout``  a differentiable trajectory of star robots and its backward pass (calibration).
* ``band``     the standalone batched banded solve.
* ``infer`` / ``train``  the warm-start network: inference on a batch of rod segments, one Adam step.

The states are smooth: every rod is a planar arc that swings at a given rate, its reference frames turned
along the rod as a simulation leaves them, so that the Newton iterations and the contacts are those of a
running simulation.
"""
import math

import numpy as np
import torch

import paper_2311_18126_gb300 as dm
from paper_2311_18126_gb300 import adjoint as dm_adjoint
from paper_2311_18126_gb300 import dismech

G = (0.0, 0.0, -9.81)
ETA = 0.1


# --------------------------------------------------------------------------------------------- cases
def listed():
    return [
        # one 50-node cantilever (L = 1 m), ten steps in a call: the smallest simulation, bound by latency
        dict(name="cantilever_10_steps", family="step", rods=1, n_min=50, n_max=50, steps=10,
             integrator="be", line_search=False),
        # the flagship batch: 4096 uneven rods of 20 to 200 nodes, backward Euler
        dict(name="rods_4096", family="step", rods=4096, n_min=20, n_max=200, steps=1,
             integrator="be", line_search=False),
        # a medium batch of odd size, implicit midpoint with the line search that stiff rods need there
        dict(name="rods_301_midpoint", family="step", rods=301, n_min=20, n_max=200, steps=1,
             integrator="midpoint", line_search=True),
        # cables: 64 rods of 4000 to 6000 nodes (the partitioned solver)
        dict(name="long_rods_64", family="step", rods=64, n_min=4000, n_max=6000, steps=1,
             integrator="be", line_search=False),
        # 1024 star robots of 3 to 8 limbs on the ground, one control step of their gait
        dict(name="star_robots_1024", family="robots", robots=1024, k_min=3, k_max=8, nodes=30),
        # a collapsed coil of 500 nodes, every turn in contact with its neighbours
        dict(name="coil_500", family="coil", nodes=500),
        # four grippers of five 60-node fingers closing on each other
        dict(name="grippers_4", family="grippers", groups=4, fingers=5, nodes=60),
        # gradients of one step of 1024 uneven rods (system identification)
        dict(name="adjoint_rods_1024", family="adjoint", rods=1024, n_min=20, n_max=200),
        # calibration: 64 four-limbed robots, six steps forward and back, a checkpoint every three
        dict(name="rollout_robots_64", family="rollout", robots=64, k_min=4, k_max=4, nodes=30, steps=6, every=3),
        # a batch of banded systems of rod size, solved for a caller that assembles its own Jacobians
        dict(name="band_1000", family="band", systems=1000, n_min=79, n_max=799),
        # network inference over the segments of the flagship batch
        dict(name="infer_444544", family="infer", rows=444544),
        # one training step of the network
        dict(name="train_16384", family="train", rows=16384),
    ]


def draw(rng):
    def logi(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["step", "step", "step", "long", "robots", "coil", "grippers", "adjoint", "rollout",
                         "band", "infer", "train"])
    if family == "step":
        lo = rng.randint(6, 60)
        return dict(family="step", rods=logi(1, 4096), n_min=lo, n_max=rng.randint(lo, 200), steps=rng.choice([1, 1, 2]),
                    integrator=rng.choice(["be", "be", "midpoint"]), line_search=True)
    if family == "long":
        lo = rng.randint(515, 4000)
        return dict(family="step", rods=rng.randint(1, 63), n_min=lo, n_max=rng.randint(lo, 6000), steps=1,
                    integrator="be", line_search=False)
    if family == "robots":
        lo = rng.randint(3, 6)
        return dict(family="robots", robots=logi(1, 1024), k_min=lo, k_max=rng.randint(lo, 8), nodes=rng.randint(20, 30))
    if family == "coil":
        return dict(family="coil", nodes=logi(120, 500))
    if family == "grippers":
        return dict(family="grippers", groups=rng.randint(1, 4), fingers=rng.randint(3, 5), nodes=rng.randint(30, 60))
    if family == "adjoint":
        lo = rng.randint(6, 60)
        return dict(family="adjoint", rods=logi(4, 2048), n_min=lo, n_max=rng.randint(lo, 200))
    if family == "rollout":
        return dict(family="rollout", robots=logi(2, 64), k_min=3, k_max=rng.randint(3, 6), nodes=rng.randint(20, 30),
                    steps=rng.randint(3, 6), every=rng.randint(2, 4))
    if family == "band":
        lo = rng.randint(11, 300)
        return dict(family="band", systems=logi(1, 4096), n_min=lo, n_max=rng.randint(lo, 799))
    if family == "infer":
        return dict(family="infer", rows=128 * logi(1, 3473))
    return dict(family="train", rows=128 * logi(4, 256))


# --------------------------------------------------------------------------------- rods as planar arcs
def _arcs(npr, spacing, base, along, into, curv, rate, spin):
    """Rods of ``npr`` nodes in the plane of the unit vectors ``along`` and ``into``: edge i at the angle
    curv * spacing * i, swinging at the rate d(curv)/dt; the reference director of each edge turned by the angle
    ``spin`` (per edge) out of the in-plane normal, the twist angle turned back by it.  Returns the state in the
    layout of the library (q, qdot) and the frames (d1 per edge, reference twist per interior node)."""
    npr = np.asarray(npr)
    q, v, d1s, betas = [], [], [], []
    for r, n in enumerate(npr):
        l, i = spacing[r], np.arange(n - 1)
        phi, dphi = curv[r] * l * i, rate[r] * l * i
        c, s = np.cos(phi)[:, None], np.sin(phi)[:, None]
        a, w = along[r][None], into[r][None]
        x = np.concatenate([np.zeros((1, 3)), np.cumsum(l * (c * a + s * w), 0)]) + base[r]
        dx = np.concatenate([np.zeros((1, 3)), np.cumsum(l * dphi[:, None] * (c * w - s * a), 0)])
        psi = spin[r][:n - 1]
        qr, vr = np.zeros(4 * n), np.zeros(4 * n)
        for k in range(3):
            qr[k::4], vr[k::4] = x[:, k], dx[:, k]
        qr[3::4][:n - 1] = -psi
        q.append(qr[:-1])
        v.append(vr[:-1])
        t, m = c * a + s * w, c * w - s * a
        d1s.append(np.cos(psi)[:, None] * m + np.sin(psi)[:, None] * np.cross(t, m))
        betas.append(np.diff(psi))
    return np.concatenate(q), np.concatenate(v), np.concatenate(d1s), np.concatenate(betas)


def _spin(rng, npr):
    """A smooth rotation of the reference frames along each rod, zero at its first edge."""
    out = []
    for n in npr:
        a, k = rng.uniform(0.2, 0.8), rng.uniform(1.0, 3.0)
        out.append(a * np.sin(k * math.pi * np.arange(n - 1) / max(n - 2, 1)))
    return out


def _clamp(npr):
    """Nodes 0 and 1 and the first twist angle of every rod fixed."""
    mask = [np.zeros(4 * n - 1, np.uint8) for n in npr]
    for m in mask:
        m[:7] = 1
    return np.concatenate(mask)


def _straight(npr, spacing, base, along):
    return np.concatenate([base[r] + np.arange(n)[:, None] * spacing[r] * along[r] for r, n in enumerate(npr)])


def _rods(case, seed):
    """(desc, params, state) of a batch of clamped rods."""
    rng = np.random.default_rng([seed, 1])
    R = case["rods"]  # the node counts are the case's: the seed draws materials, shapes and motion
    npr = np.random.default_rng([R, case["n_min"], case["n_max"]]).integers(case["n_min"], case["n_max"] + 1, R)
    if R == 1:  # the cantilever: 1 m, h = 1 mm, E = 1e7
        L, h, E = np.ones(1), np.full(1, 1e-3), np.full(1, 1e7)
    else:
        L, h, E = rng.uniform(0.2, 1.5, R), rng.uniform(5e-4, 3e-3, R), 10.0 ** rng.uniform(6.0, 8.0, R)
    if case["n_max"] > 500:  # cables: the edge length stays that of the short rods
        L = L * npr / 110.0
    spacing = L / (npr - 1)
    ang = rng.uniform(0.0, 2.0 * math.pi, R)
    base = rng.uniform(-0.1, 0.1, (R, 3))  # every rod in a frame of its own: they do not see each other
    along = np.stack([np.cos(ang), np.sin(ang), np.zeros(R)], 1)
    into = np.tile([0.0, 0.0, 1.0], (R, 1))
    c1, c2 = rng.uniform(-5.0, 5.0, (2, R)) / np.maximum(1.0, L / 1.5)
    curv, rate = c1 * rng.uniform(0.3, 0.9, R), np.abs(c1) * rng.uniform(-0.5, 0.5, R)
    q, v, d1, beta = _arcs(npr, spacing, base, along, into, curv, rate, _spin(rng, npr))
    desc = dict(nodes_per_rod=npr.astype(np.int32), x0=_straight(npr, spacing, base, along), E=E, nu=np.full(R, 0.5),
                rho=np.full(R, 1000.0), radius=h, fixed=_clamp(npr))
    params = dict(dt=1e-3, tol=1e-10, max_iter=100, g=G, eta=ETA, line_search=case.get("line_search", False),
                  integrator=case.get("integrator", "be"), predictor="projected")
    kbar = np.concatenate([np.tile([c1[r] * spacing[r], c2[r] * spacing[r]], (n - 2, 1)) for r, n in enumerate(npr)])
    return desc, params, (q, v, d1, beta, kbar)


def _robots(case, seed, times=1):
    """Star robots: limbs joined at a centre node, lying on the ground, the limbs of positive natural curvature
    curled up; ``times`` rows of natural curvatures of consecutive steps."""
    rng = np.random.default_rng([seed, 2])
    B, N, dt = case["robots"], case["nodes"], 5e-3
    h, delta, length = 2e-3, 5e-4, 0.1
    ks = np.random.default_rng([B, case["k_min"], case["k_max"]]).integers(case["k_min"], case["k_max"] + 1, B)
    amp, per, mu = rng.uniform(0.0, 20.0, B), rng.uniform(0.5, 2.0, B), rng.uniform(0.3, 0.8, B)
    t0, frac = rng.uniform(0.0, 2.0, B), rng.uniform(0.3, 0.6, B)
    l = length / (N - 1)
    kc = 50.0 * 1000.0 * math.pi * h * h * l * 9.81 / delta
    bot = np.repeat(np.arange(B), ks)
    j = np.concatenate([np.arange(k) for k in ks])
    R = len(bot)
    a = 2.0 * math.pi * j / ks[bot]
    centre = rng.uniform(-0.1, 0.1, (B, 2))
    base = np.concatenate([centre[bot], np.full((R, 1), h)], 1)
    along = np.stack([np.cos(a), np.sin(a), np.zeros(R)], 1)
    into = np.tile([0.0, 0.0, 1.0], (R, 1))

    def curvature(step):
        return amp[bot] * np.sin(2.0 * math.pi * (t0[bot] + (step + 1) * dt) / per[bot] + a)

    npr = np.full(R, N)
    curv = np.maximum(curvature(-1), 0.0) * frac[bot]
    rest = np.array([0.0, 0.0, 0.05 * delta])  # where the contact force carries the weight
    spin = _spin(rng, npr)
    q, v, d1, beta = _arcs(npr, np.full(R, l), base + rest, along, into, curv, 0.1 * curv, spin)
    # reference twists by node: per robot the pairs at its centre, then its limbs
    inner, at = beta.reshape(R, N - 2), np.concatenate([[0], np.cumsum(ks)])
    beta = np.concatenate([np.concatenate([np.zeros(k * (k - 1) // 2), inner[at[b]:at[b + 1]].reshape(-1)])
                           for b, k in enumerate(ks)])
    desc = dict(nodes_per_rod=npr.astype(np.int32), x0=_straight(npr, np.full(R, l), base, along), E=np.full(R, 1e6),
                nu=np.full(R, 0.5), rho=np.full(R, 1000.0), radius=np.full(R, h),
                fixed=np.zeros(R * (4 * N - 1), np.uint8),
                joints=[[(int(at[b]) + i, 0) for i in range(k)] for b, k in enumerate(ks)],
                ground_mu=mu[bot], ground_kc=np.full(R, kc))
    params = dict(dt=dt, tol=1e-10, max_iter=100, g=G, eta=ETA, ground=True, ground_z=0.0, delta=delta, nu_slip=1e-3,
                  line_search=True)
    kbar = np.zeros((times, R, N - 2, 2))
    for s in range(times):
        kbar[s, :, :, 0] = (curvature(s) * l)[:, None]
    return desc, params, (q, v, d1, beta, kbar.reshape(times, -1, 2))


def _coil(case, seed):
    """A helix of radius 2 cm, stress-free at a pitch of 2.2 radii, collapsed until the turns touch."""
    rng = np.random.default_rng([seed, 3])
    N, h, radius, spacing, delta, E = case["nodes"], 1e-3, 0.02, 2.5e-3, 1e-4, 1e7
    turn = math.hypot(2.0 * math.pi * radius, 2.2 * h)
    phi = 2.0 * math.pi * np.arange(N) * spacing / turn

    def helix(pitch):
        return np.stack([radius * np.cos(phi), radius * np.sin(phi), pitch * phi / (2.0 * math.pi)], 1)

    fixed = _clamp([N])
    x = helix(h * rng.uniform(2.04, 2.08))
    x[:, 2] += 5e-6 * np.sin(phi * rng.uniform(0.2, 0.7)) * (phi / phi[-1])
    vel = np.zeros((N, 3))
    vel[2:, 2] = -rng.uniform(0.01, 0.02) * (phi / phi[-1])[2:]
    q, v = np.zeros(4 * N), np.zeros(4 * N)
    for k in range(3):
        q[k::4], v[k::4] = x[:, k], vel[:, k]
    psi = _spin(rng, [N])[0]
    q[3::4][:N - 1] = -psi
    desc = dict(nodes_per_rod=np.array([N], np.int32), x0=helix(2.2 * h), E=np.array([E]), nu=np.array([0.5]),
                rho=np.array([1000.0]), radius=np.array([h]), fixed=fixed)
    params = dict(dt=2.5e-4, tol=1e-10, max_iter=100, g=G, eta=ETA, self_contact=True, delta=delta, pair_kc=E * h,
                  pair_mu=0.0, line_search=True)
    return desc, params, (q[:-1], v[:-1], (x, psi))


def _grippers(case, seed):
    """Grippers: fingers hanging from a ring of 3 cm, curled inwards until neighbouring tips touch."""
    rng = np.random.default_rng([seed, 4])
    B, F, N = case["groups"], case["fingers"], case["nodes"]
    h, delta, E, ring, l = 2.5e-3, 5e-4, 3e5, 0.03, 0.3 / 59
    R = B * F
    a = 2.0 * math.pi * (np.arange(R) % F) / F
    radial = np.stack([np.cos(a), np.sin(a), np.zeros(R)], 1)
    base = ring * radial
    along = np.tile([0.0, 0.0, -1.0], (R, 1))
    reach = ring - 0.5 * (2.0 * h + 0.5 * delta) / math.sin(math.pi / F)

    def inward(c):  # of the last node
        return l * np.sin(c * l * np.arange(N - 1)).sum()

    lo, hi = 0.0, 0.5 * math.pi / (l * (N - 1))
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if inward(mid) < reach else (lo, mid)
    curv = lo * rng.uniform(0.998, 1.002, R)
    npr = np.full(R, N)
    spacing = np.full(R, l)
    q, v, d1, beta = _arcs(npr, spacing, base, along, -radial, curv, rng.uniform(0.3, 0.6, R) * curv, _spin(rng, npr))
    desc = dict(nodes_per_rod=npr.astype(np.int32), x0=_straight(npr, spacing, base, along), E=np.full(R, E),
                nu=np.full(R, 0.5), rho=np.full(R, 1200.0), radius=np.full(R, h), fixed=_clamp(npr),
                contact_groups=[list(range(F * b, F * b + F)) for b in range(B)])
    params = dict(dt=1e-3, tol=1e-10, max_iter=100, g=G, eta=ETA, self_contact=True, delta=delta, pair_kc=E * h,
                  pair_mu=0.5, nu_slip=1e-3, line_search=True)
    kbar = np.zeros((R, N - 2, 2))
    kbar[:, :, 0] = (curv * l * rng.uniform(1.0, 1.3, R))[:, None]
    return desc, params, (q, v, d1, beta, kbar.reshape(-1, 2))


# ------------------------------------------------------------------------------------ the other inputs
def _band(case, seed):
    """Symmetric positive definite band matrices (half bandwidth 10) B B^T of uneven systems: band [11, n], rhs."""
    rng = np.random.default_rng([seed, 5])
    sizes = np.random.default_rng([case["systems"], case["n_min"], case["n_max"]])
    ndof = sizes.integers(case["n_min"], case["n_max"] + 1, case["systems"])
    dof0 = np.concatenate([[0], np.cumsum(ndof)])
    n = int(dof0[-1])
    row = np.arange(n) - np.repeat(dof0[:-1], ndof)
    B = rng.normal(0.0, 0.2, (11, n))
    B[0] = 10.0 ** rng.uniform(0.0, 1.0, n)
    for m in range(11):
        B[m, row < m] = 0.0
    band = np.zeros((11, n))
    for d in range(11):
        for m in range(d, 11):
            band[d, d:] += B[m, d:] * B[m - d, :n - d]
        band[d, row < d] = 0.0
    return dof0[:-1].astype(np.int32), ndof.astype(np.int32), band, rng.normal(0.0, 1.0, n)


N_IN, N_OUT = 61, 4
SHAPES = [(256, 64), (256, 256), (256, 256), (64, 256)]


def _network(seed):
    """Parameters in the library's layout: per layer W [out][in], b [out], unused inputs and outputs zero."""
    rng = np.random.default_rng([seed, 6])
    out = []
    for k, (o, i) in enumerate(SHAPES):
        W = rng.normal(0.0, math.sqrt(2.0 / (N_IN if k == 0 else i)), (o, i))
        b = rng.normal(0.0, 0.05, o)
        if k == 0:
            W[:, N_IN:] = 0.0
        if k == 3:
            W[N_OUT:], b[N_OUT:] = 0.0, 0.0
        out += [W.reshape(-1), b]
    return np.concatenate(out).astype(np.float32)


def _rows(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((case["rows"], 64), generator=g, device="cuda")
    X[:, N_IN:] = 0.0
    Y = torch.randn((case["rows"], N_OUT), generator=g, device="cuda")
    return X.to(torch.bfloat16), Y


# --------------------------------------------------------------------------------------- prepare, run
def _gpu(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).cuda()


def prepare(case, seed):
    family = case["family"]
    s = dict(family=family)
    if family == "band":
        dof0, ndof, band, rhs = _band(case, seed)
        s.update(dof0=dof0, ndof=ndof, band=_gpu(band), rhs=_gpu(rhs), x=torch.empty(len(rhs), dtype=torch.float64).cuda())
        return s
    if family in ("infer", "train"):
        X, Y = _rows(case, seed)
        net = dismech.MLP(N_IN, N_OUT, seed=0)
        net.set_params(_network(seed))
        s.update(net=net, X=X, Y=Y)
        if family == "infer":
            s["out"] = torch.empty((case["rows"], 64), dtype=torch.float32, device="cuda")
        else:
            s["grads"] = torch.empty(net.n_params, dtype=torch.float32, device="cuda")
        return s
    if family in ("step", "adjoint"):
        desc, params, (q, v, d1, beta, kbar) = _rods(case, seed)
    elif family == "robots":
        desc, params, (q, v, d1, beta, kbar) = _robots(case, seed)
        kbar = kbar[0]
    elif family == "rollout":
        desc, params, (q, v, d1, beta, kbar) = _robots(case, seed, case["steps"])
    elif family == "coil":
        desc, params, (q, v, turned) = _coil(case, seed)
    else:
        desc, params, (q, v, d1, beta, kbar) = _grippers(case, seed)
    system = dm.System(desc, params)
    if family == "coil":  # natural curvatures are those of the rest shape; the frames follow the turned edges
        x, psi = turned
        d1, beta = system.get_frames()
        t = np.diff(x, axis=0)
        t /= np.linalg.norm(t, axis=1)[:, None]
        d1 = d1 - (d1 * t).sum(1)[:, None] * t
        d1 /= np.linalg.norm(d1, axis=1)[:, None]
        d1 = np.cos(psi)[:, None] * d1 + np.sin(psi)[:, None] * np.cross(t, d1)
        beta, kbar = beta + np.diff(psi), None
    s.update(system=system, steps=case.get("steps", 1), q=_gpu(q), v=_gpu(v), d1=_gpu(d1), beta=_gpu(beta),
             kbar=None if kbar is None else _gpu(kbar))
    if family == "rollout":
        rng = np.random.default_rng([seed, 7])
        for k in ("kbar", "q", "v"):
            s[k].requires_grad_(True)
        s.update(every=case["every"], frames=(d1, beta), grad=_gpu(rng.normal(0.0, 1.0, (case["steps"], len(q)))))
    else:
        s["out"] = [torch.empty_like(s[k]) for k in ("q", "v", "d1", "beta")]
    if family == "adjoint":  # the step whose adjoint is taken, then back to its start
        rng = np.random.default_rng([seed, 7])
        s.update(gq=_gpu(rng.normal(0.0, 1.0, len(q))), gv=_gpu(rng.normal(0.0, 1e-3, len(q))))
        s["next"] = _step(s)[0].clone()
        system.set_state(s["q"], s["v"])
        system.set_frames(s["d1"], s["beta"])
    torch.cuda.synchronize()
    return s


def _step(s):
    system = s["system"]
    system.set_state(s["q"], s["v"])
    system.set_frames(s["d1"], s["beta"])
    if s["kbar"] is not None:
        system.set_natural_curvature(0, system.n_rods, s["kbar"])
    system.step(s["steps"], stats=False)
    q, v, d1, beta = s["out"]
    system.get_state(q, v)
    system.get_frames(d1, beta)
    return s["out"]


def run(s):
    family = s["family"]
    if family == "band":
        return dismech.solve_band(s["dof0"], s["ndof"], s["band"], s["rhs"], s["x"])
    if family == "infer":
        return s["net"].forward_async(s["X"], s["out"])
    if family == "train":
        loss = s["net"].train_step(s["X"], s["Y"], 1e-3, s["grads"])
        return loss, s["grads"]
    if family == "adjoint":
        return s["system"].step_adjoint(s["next"], s["gq"], s["gv"])
    if family == "rollout":
        x = dm_adjoint.rollout(s["system"], s["kbar"], s["q"], s["v"], s["frames"], s["every"])
        return (x.detach(),) + torch.autograd.grad(x, [s["kbar"], s["q"], s["v"]], s["grad"])
    return _step(s)


# ------------------------------------------------------------------------------------------------ work
def work(case):
    """Bytes of the inputs and outputs, and the operations of a pass: per Newton iteration about 2000 per
    bend-twist stencil with its edge and 160 per DOF of the band factorisation, two iterations a step."""
    family = case["family"]
    if family == "band":
        n = case["systems"] * 0.5 * (case["n_min"] + case["n_max"])
        return dict(bytes=13 * 8 * n, flops=160 * n)
    if family in ("infer", "train"):
        params = sum(o * i + o for o, i in SHAPES)
        flops = 2.0 * case["rows"] * sum(o * i for o, i in SHAPES)
        if family == "infer":
            return dict(bytes=case["rows"] * (128 + 256) + 4 * params, flops=flops)
        return dict(bytes=case["rows"] * (128 + 16) + 4 * 8 * params, flops=3 * flops)
    if family in ("step", "adjoint"):
        nodes = case["rods"] * 0.5 * (case["n_min"] + case["n_max"])
    elif family in ("robots", "rollout"):
        nodes = case["robots"] * 0.5 * (case["k_min"] + case["k_max"]) * case["nodes"]
    elif family == "coil":
        nodes = case["nodes"]
    else:
        nodes = case["groups"] * case["fingers"] * case["nodes"]
    per_iteration = (2000 + 4 * 160) * nodes
    if family in ("coil", "grippers"):  # a dense elimination of each system of touching rods
        n = 4.0 * nodes / case.get("groups", 1)
        per_iteration += case.get("groups", 1) * 2.0 / 3.0 * n ** 3 / 8
    state = 8 * nodes * (8 + 3 + 1)  # q, qdot, director, reference twist
    if family == "adjoint":
        return dict(bytes=8 * nodes * (4 * 5 + 2), flops=per_iteration)
    steps = case.get("steps", 1)
    if family == "rollout":  # forward, once more for the segments, the adjoint of each step
        return dict(bytes=steps * 8 * nodes * (4 + 4 + 2 + 2), flops=steps * 5 * per_iteration)
    return dict(bytes=2 * state + 16 * nodes, flops=steps * 2 * per_iteration)


# ----------------------------------------------------------------------------------------------- exact
# Clamped rods in 64 bits, from the energies by automatic differentiation: one implicit step of a batch.
def _turn(u, a, b):
    """u carried from the unit vector a to the unit vector b by the least rotation."""
    w = torch.linalg.cross(a, b)
    return u * a.dot(b) + torch.linalg.cross(w, u) + w * (w.dot(u) / (1.0 + a.dot(b)))


def _stencil_energy(z, c):
    """Bending and twisting energy of two edges: z = x0 th0 x1 th1 x2 (11); c: tangents and directors of the
    committed step (12), its reference twist, EI/V, GJ/V, the natural curvatures (2)."""
    D, T = [], []
    for e in range(2):
        d = z[4 * e + 4:4 * e + 7] - z[4 * e:4 * e + 3]
        T.append(d / d.dot(d).sqrt())
        D.append(_turn(c[6 + 3 * e:9 + 3 * e], c[3 * e:3 * e + 3], T[e]))
    m1 = [torch.cos(z[4 * e + 3]) * D[e] + torch.sin(z[4 * e + 3]) * torch.linalg.cross(T[e], D[e]) for e in range(2)]
    m2 = [torch.linalg.cross(T[e], m1[e]) for e in range(2)]
    kb = 2.0 * torch.linalg.cross(T[0], T[1]) / (1.0 + T[0].dot(T[1]))
    k1, k2 = 0.5 * kb.dot(m2[0] + m2[1]), -0.5 * kb.dot(m1[0] + m1[1])
    w = _turn(D[0], T[0], T[1])
    beta = torch.atan2(torch.linalg.cross(w, D[1]).dot(T[1]), w.dot(D[1]))
    beta = beta + 2.0 * math.pi * torch.round((c[12] - beta.detach()) / (2.0 * math.pi))
    tw = z[7] - z[3] + beta
    return 0.5 * c[13] * ((k1 - c[15]) ** 2 + (k2 - c[16]) ** 2) + 0.5 * c[14] * tw ** 2, beta


def _stretch_energy(z, c):
    d = z[3:6] - z[0:3]
    return 0.5 * c[0] * c[1] * (d.dot(d).sqrt() / c[1] - 1.0) ** 2


class _Rods:
    """The batch on a grid of 4 DOFs per node: DOF 4 n + c, nodes of the rods one after another."""

    def __init__(self, case, seed):
        desc, self.params, (q, v, d1, beta, kbar) = _rods(case, seed)
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
        npr = np.asarray(desc["nodes_per_rod"], np.int64)
        R, n0 = len(npr), np.concatenate([[0], np.cumsum(npr)])
        rod = np.repeat(np.arange(R), npr)
        i = np.arange(n0[-1]) - n0[rod]
        last = i == npr[rod] - 1
        lay = np.flatnonzero(~((np.arange(4 * n0[-1]) % 4 == 3) & np.repeat(last, 4)))  # grid place of each layout entry
        self.n, self.lay = 4 * int(n0[-1]), T(lay)
        self.edge, self.mid = T(np.flatnonzero(~last)), T(np.flatnonzero(~last & (i > 0)))
        x = desc["x0"]
        l = np.zeros(n0[-1])
        l[~last] = np.linalg.norm(x[1:] - x[:-1], axis=1)[~last[:-1]]
        before = np.concatenate([[0.0], l[:-1]])  # a rod's last node has no edge: l = 0 there
        area, E, h = math.pi * desc["radius"] ** 2, desc["E"], desc["radius"]
        GS = E / (2.0 * (1.0 + desc["nu"]))
        V = 0.5 * (l + before)
        mass = np.zeros((n0[-1], 4))
        mass[:, :3] = (desc["rho"] * area)[rod, None] * V[:, None]
        mass[:, 3] = (desc["rho"] * area * h * h / 2.0)[rod] * l
        self.mass, self.damp = T(mass.reshape(-1)), T(np.repeat(ETA * V, 4) * np.tile([1.0, 1.0, 1.0, 0.0], n0[-1]))
        self.grav = self.mass * T(np.tile([*self.params["g"], 0.0], n0[-1]))
        fixed = np.ones(self.n, bool)
        fixed[lay] = desc["fixed"].astype(bool)
        self.free = T(~fixed)
        self.EA, self.l = T((E * area)[rod])[self.edge], T(l)[self.edge]
        m = self.mid.cpu().numpy()
        EI, GJ = E * math.pi * h ** 4 / 4.0, GS * math.pi * h ** 4 / 2.0
        self.coef = T(np.stack([EI[rod][m] / V[m], GJ[rod][m] / V[m], kbar[:, 0], kbar[:, 1]], 1))
        self.eid = torch.zeros(int(n0[-1]), dtype=torch.int64, device="cuda")
        self.eid[self.edge] = torch.arange(len(self.edge), device="cuda")
        self.rod = T(np.repeat(rod, 4))
        # blocks of three nodes per rod for the elimination
        self.R, self.nb = R, int((npr.max() + 2) // 3)
        place = T(np.repeat(rod * self.nb * 12 + 4 * i, 4) + np.tile(np.arange(4), n0[-1]))
        self.place = place
        self.grid = lambda a: torch.zeros(self.n, dtype=torch.float64, device="cuda").index_copy(0, self.lay, T(a))
        self.q0, self.v0, self.d1, self.beta0 = self.grid(q), self.grid(v), T(d1), T(beta)

    def tangents(self, q):
        x = q.view(-1, 4)[:, :3]
        d = x[self.edge + 1] - x[self.edge]
        return d / d.norm(dim=1, keepdim=True)

    def commit(self, qn, d1, beta):
        t = self.tangents(qn)
        a, b = self.eid[self.mid - 1], self.eid[self.mid]
        self.c = torch.cat([t[a], t[b], d1[a], d1[b], beta[:, None], self.coef], 1)
        self.sidx = 4 * (self.mid[:, None] - 1) + torch.arange(11, device="cuda")
        self.tidx = 4 * self.edge[:, None] + torch.tensor([0, 1, 2, 4, 5, 6], device="cuda")
        self.sc = torch.stack([self.EA, self.l], 1)

    def forces(self, q, hess):
        """dE/dq, and the element Hessians [(index, matrices)] on request."""
        f, H = torch.zeros_like(q), []
        for fun, idx, c in ((lambda z, c: _stencil_energy(z, c)[0], self.sidx, self.c), (_stretch_energy, self.tidx, self.sc)):
            vg, vh = torch.func.vmap(torch.func.grad(fun)), torch.func.vmap(torch.func.hessian(fun))
            Hs = []
            for at in range(0, len(idx), 100000):
                z, cc = q[idx[at:at + 100000]], c[at:at + 100000]
                f.index_add_(0, idx[at:at + 100000].reshape(-1), vg(z, cc).reshape(-1))
                if hess:
                    Hs.append(vh(z, cc))
            if hess:
                H.append((idx, torch.cat(Hs)))
        return (f, H) if hess else f

    def solve(self, diag, H, rhs):
        """(diag + sum of H) x = rhs on the free DOFs, block tridiagonal elimination per rod."""
        R, nb = self.R, self.nb
        A = torch.zeros(R * nb * 3 * 144, dtype=torch.float64, device="cuda")
        put = lambda i, j, v: A.index_add_(0, ((i // 12) * 3 + (j // 12 - i // 12) + 1) * 144 + (i % 12) * 12 + j % 12, v)  # noqa: E731
        used = torch.zeros(R * nb * 12, dtype=torch.bool, device="cuda")
        used[self.place] = self.free
        every = torch.arange(R * nb * 12, device="cuda")
        d = torch.ones(R * nb * 12, dtype=torch.float64, device="cuda")
        d[self.place[self.free]] = diag[self.free]
        put(every, every, d)
        for idx, h in H:
            ok = (self.free[idx][:, :, None] & self.free[idx][:, None, :]).reshape(-1)
            i = self.place[idx][:, :, None].expand_as(h).reshape(-1)[ok]
            j = self.place[idx][:, None, :].expand_as(h).reshape(-1)[ok]
            put(i, j, h.reshape(-1)[ok])
        A = A.view(R, nb, 3, 12, 12)
        b = torch.zeros(R * nb * 12, dtype=torch.float64, device="cuda")
        b[self.place] = torch.where(self.free, rhs, torch.zeros_like(rhs))
        x = _tridiagonal(A, b.view(R, nb, 12))
        return x.reshape(-1)[self.place] * self.free

    def step(self):
        """q, qdot, d1, beta after one step."""
        mid = self.params["integrator"] == "midpoint"
        h = self.params["dt"] * (0.5 if mid else 1.0)
        qn, vn = self.q0, self.v0
        self.commit(qn, self.d1, self.beta0)
        diag = self.mass / h ** 2 + self.damp / h

        def residual(q, hess):
            f = self.forces(q, hess)
            f, H = f if hess else (f, None)
            f = f + self.mass * ((q - qn) / h - vn) / h + self.damp * (q - qn) / h - self.grav
            return torch.where(self.free, f, torch.zeros_like(f)), H

        def merit(f):
            return torch.zeros(self.R, dtype=torch.float64, device="cuda").index_add_(0, self.rod, (f / diag.clamp_min(1e-300)) ** 2)

        y = torch.where(self.free, qn + h * vn, qn)
        f, H = residual(y, True)
        for _ in range(40):
            dq, was = self.solve(diag, H, -f), merit(f)
            step = torch.ones(self.R, dtype=torch.float64, device="cuda")
            for _ in range(10):
                z = y + step[self.rod] * dq
                g = merit(residual(z, False)[0])
                worse = (g > was) & (g > 1e-24 * self.R)
                if not bool(worse.any()):
                    break
                step[worse] *= 0.5
            moved = float((step[self.rod] * dq).abs().max())
            y = y + step[self.rod] * dq
            f, H = residual(y, True)
            if moved < 1e-13:
                break
        self.y, self.H, self.diag, self.h = y, H, diag, h
        q1 = 2.0 * y - qn if mid else y
        v1 = 2.0 * (q1 - qn) / self.params["dt"] - vn if mid else (q1 - qn) / h
        q1, v1 = torch.where(self.free, q1, qn), torch.where(self.free, v1, torch.zeros_like(v1))
        ta, tb = self.tangents(qn), self.tangents(q1)
        d1 = torch.func.vmap(_turn)(self.d1, ta, tb)
        d1 = d1 / d1.norm(dim=1, keepdim=True)
        beta = torch.func.vmap(lambda z, c: _stencil_energy(z, c)[1])(q1[self.sidx], self.c)
        return q1, v1, d1, beta

    def adjoint(self, gq, gv):
        """Gradients of gq . q_{n+1} + gv . qdot_{n+1}: natural curvatures, q_n, qdot_n (backward Euler, the committed
        frames held; fixed DOFs pass theirs through)."""
        self.step()
        gq, gv, h = self.grid(gq), self.grid(gv), self.h
        lam = self.solve(self.diag, self.H, gq + gv / h)

        def pulled(k, z, c, w):  # w . d(dE/dz) for the natural curvatures k
            return torch.func.grad(lambda u: _stencil_energy(u, torch.cat([c[:15], k]))[0])(z).dot(w)

        z = self.y[self.sidx]
        gk = -torch.func.vmap(torch.func.grad(pulled))(self.c[:, 15:], z, self.c, lam[self.sidx])
        gq0 = torch.where(self.free, lam * (self.mass / h ** 2 + self.damp / h) - gv / h, gq)
        gv0 = torch.where(self.free, lam * self.mass / h, torch.zeros_like(lam))
        return gk, gq0[self.lay], gv0[self.lay]


def _tridiagonal(A, b):
    """Block tridiagonal systems A [R, nb, 3, m, m] (blocks left, middle, right), b [R, nb, m]."""
    nb = A.shape[1]
    C, y = [], []
    for k in range(nb):
        M, r = A[:, k, 1], b[:, k, :, None]
        if k:
            M = M - A[:, k, 0] @ C[-1]
            r = r - A[:, k, 0] @ y[-1]
        s = torch.linalg.solve(M, torch.cat([A[:, k, 2], r], 2))
        C.append(s[:, :, :-1])
        y.append(s[:, :, -1:])
    x = [y[-1]]
    for k in range(nb - 2, -1, -1):
        x.append(y[k] - C[k] @ x[-1])
    return torch.cat(x[::-1], 2).transpose(1, 2).contiguous()


def _exact_band(case, seed):
    dof0, ndof, band, rhs = _band(case, seed)
    R, nb = len(ndof), int((ndof.max() + 11) // 12)
    A = np.zeros((R, nb, 3, 12, 12))
    sysid = np.repeat(np.arange(R), ndof)
    i = np.arange(len(rhs)) - np.repeat(dof0, ndof)
    A[:, :, 1, range(12), range(12)] = 1.0
    for d in range(11):
        ok = i >= d
        a, r, c = sysid[ok], i[ok], i[ok] - d
        A[a, r // 12, c // 12 - r // 12 + 1, r % 12, c % 12] = band[d, ok]
        A[a, c // 12, r // 12 - c // 12 + 1, c % 12, r % 12] = band[d, ok]
    b = np.zeros((R, nb * 12))
    b[sysid, i] = rhs
    x = _tridiagonal(torch.as_tensor(A).cuda(), torch.as_tensor(b).cuda().view(R, nb, 12))
    return x.reshape(R, -1)[torch.as_tensor(sysid).cuda(), torch.as_tensor(i).cuda()]


def _forward(params, X):
    h, at = X, 0
    for k, (o, i) in enumerate(SHAPES):
        W, b = params[at:at + o * i].view(o, i), params[at + o * i:at + o * i + o]
        at += o * i + o
        h = h @ W.T + b
        h = h.relu() if k < 3 else h
    return h


def exact(case, seed):
    family = case["family"]
    if family == "band":
        return _exact_band(case, seed)
    if family in ("infer", "train"):
        X, Y = _rows(case, seed)
        p = torch.as_tensor(_network(seed)).cuda().double()
        if family == "infer":
            return _forward(p, X.double())
        p.requires_grad_(True)
        loss = ((_forward(p, X.double())[:, :N_OUT] - Y.double()) ** 2).mean()
        return float(loss.detach()), torch.autograd.grad(loss, p)[0]
    if family == "adjoint":
        rods = _Rods(case, seed)
        rng = np.random.default_rng([seed, 7])
        return rods.adjoint(rng.normal(0.0, 1.0, len(rods.lay)), rng.normal(0.0, 1e-3, len(rods.lay)))
    if family == "step" and case["steps"] <= 10 and case["rods"] * case["n_max"] * case["steps"] < 1_000_000:
        rods = _Rods(case, seed)
        for _ in range(case["steps"]):
            q, v, d1, beta = rods.step()
            rods.q0, rods.v0, rods.d1, rods.beta0 = q, v, d1, beta
        return q[rods.lay], v[rods.lay], d1, beta
    # joints, ground and edge-edge contact: Newton with a contact search and dense matrices in plain torch takes minutes
    return None
