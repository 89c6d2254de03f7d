"""The work whose speed this library is judged by: what a program that trains and evaluates drone
policies has it do, through the public entry points of the Python package.

Kinds of case, and what each stands for:
  step        a policy loop: control steps with observations, one call per step; eager for the
              smallest swarm (latency), replayed from a CUDA graph for the others
  rollout     K control steps in one persistent launch, with observations after every step (an
              experience buffer) or after the last one; uniform or uneven environment sizes
  render      the camera frames of every drone (colour and segmentation; depth is left out, since
              a silhouette pixel that rounds to the other side turns a number into an infinity)
  network     the surrogate network's forward pass over a batch of standardised rows
  surrogate   a control step with the surrogate in place of the integrator
  train       minibatch training steps of the surrogate: gradients and Adam
  transition  one recorded transition of the plain integrator (inputs, step, state change)
  dataset     the standardisation of a set of transitions for training

Sizes are those of the repository's own workloads (64 x 1, 16384 x 4, 1024 x 64, 4096 uneven
environments, 262144 surrogate rows, batches of 8192) and odd neighbours of them. Swarms start in
formations whose drones fly on height levels of their own, with RPM actions near hover or waypoints
that shift the formation: the downwash law diverges as 1 / dz^2, and two correct implementations
part within a few substeps where two drones of one column pass through the same height.

`exact` restates every path in float64 torch, from the equations alone.
"""
import math

import numpy as np
import torch

import paper_2606_08039_gb300 as mdg
from paper_2606_08039_gb300 import workloads as wl

DEV = "cuda"
SUBSTEPS = 5
UNEVEN_SIZES = (1, 2, 4, 8, 16, 32)
GND, DRAG, DW = 1, 2, 4


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest loop: 64 single drones, a policy that sets motor speeds, eager calls
        dict(name="single", kind="step", envs=64, drones=1, action="rpm", integrator="euler", steps=8, graph=False,
             randomize=False),
        # the headline workload: 16384 environments of 4 drones under the waypoint controller
        dict(name="full_aero", kind="step", envs=16384, drones=4, action="pid", integrator="euler", steps=8, graph=True,
             randomize=False),
        # dense swarms: 63 downwash pairs and a 64-drone neighbour search per drone
        dict(name="dense", kind="step", envs=1024, drones=64, action="rpm", integrator="euler", steps=4, graph=True,
             randomize=False),
        # training under domain randomization, motor lag, latency, wind and sensor noise
        dict(name="randomized", kind="step", envs=16384, drones=4, action="pid", integrator="euler", steps=8,
             graph=True, randomize=True),
        # mixed sizes, physics subsets and action types in one persistent launch
        dict(name="uneven_rollout", kind="rollout", envs=4096, drones=0, action="mixed", steps=32, every=False),
        # an experience buffer: every step's observations of the headline swarm
        dict(name="episode_rollout", kind="rollout", envs=16384, drones=4, action="pid", steps=32, every=True),
        # camera observations
        dict(name="camera", kind="render", envs=4099, drones=4),
        # the surrogate network over the evaluation swarm's rows
        dict(name="network", kind="network", rows=262144),
        # surrogate control steps; the drone count is no multiple of the network's row tile
        dict(name="surrogate", kind="surrogate", envs=50001, drones=4, action="pid"),
        # four minibatches of surrogate training
        dict(name="train", kind="train", batch=8192, batches=4),
        # training data of the dense Runge-Kutta swarm, the one where the surrogate pays off
        dict(name="transition", kind="transition", envs=1024, drones=64, integrator="rk4"),
        # two million transitions standardised for training
        dict(name="dataset", kind="dataset", rows=2000003),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "randomized", "rollout", "render", "network", "surrogate", "train", "transition",
                       "dataset"])
    drones = rng.choice([1, 2, 3, 4, 4, 5, 6, 7, 8, 13, 16, 30, 32, 64])
    if kind in ("step", "randomized"):
        dr = kind == "randomized"
        return dict(kind="step", envs=max(1, _log(rng, 64, 65536) // drones), drones=drones,
                    action=rng.choice(["rpm", "pid", "vel", "attitude"]),
                    integrator="euler" if dr else rng.choice(["euler", "euler", "rk4"]), steps=rng.choice([1, 2, 4, 8]),
                    graph=rng.random() < 0.5, randomize=dr)
    if kind == "rollout":
        if rng.random() < 0.5:
            return dict(kind=kind, envs=_log(rng, 64, 4096), drones=0, action="mixed", steps=rng.randint(4, 32),
                        every=rng.random() < 0.5)
        return dict(kind=kind, envs=max(1, _log(rng, 256, 65536) // drones), drones=drones,
                    action=rng.choice(["rpm", "pid"]), steps=rng.randint(4, 32), every=rng.random() < 0.5)
    if kind == "render":
        return dict(kind=kind, envs=max(1, _log(rng, 64, 16384) // drones), drones=drones)
    if kind == "network":
        return dict(kind=kind, rows=128 * _log(rng, 8, 2048))
    if kind == "surrogate":
        return dict(kind=kind, envs=max(1, _log(rng, 1024, 200000) // drones), drones=drones,
                    action=rng.choice(["rpm", "pid"]))
    if kind == "train":
        return dict(kind=kind, batch=128 * _log(rng, 8, 64), batches=rng.randint(1, 4))
    if kind == "transition":
        return dict(kind=kind, envs=max(1, _log(rng, 1024, 65536) // drones), drones=drones,
                    integrator=rng.choice(["euler", "rk4"]))
    return dict(kind="dataset", rows=_log(rng, 50000, 2000003))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _u(g, shape, lo, hi):
    """U[lo, hi) in float64, rounded to float32 values (what both sides consume)."""
    return (lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)).float().double()


def _quat(rpy):
    (sr, sp, sy), (cr, cp, cy) = torch.sin(rpy / 2).unbind(-1), torch.cos(rpy / 2).unbind(-1)
    return torch.stack([cr * cp * cy + sr * sp * sy, sr * cp * cy - cr * sp * sy, cr * sp * cy + sr * cp * sy,
                        cr * cp * sy - sr * sp * cy], -1)


def _formation(E, N, g, yaw=0.1):
    """E formations of N drones on a grid, every drone on a height level of its own. The levels of the
    small ones widen upwards, so that a drone's neighbours are at clearly different distances."""
    side = math.ceil(math.sqrt(N))
    small = N <= 8
    px, py, level, jitter = (0.25, 0.4, 0.3, 0.02) if small else (0.6, 0.6, 0.15, 0.05)
    k = torch.arange(N, device=DEV, dtype=torch.float64)
    nominal = torch.stack([(torch.remainder(k, side) - (side - 1) / 2) * px,
                           (torch.floor(k / side) - (side - 1) / 2) * py,
                           0.4 + level * k + (0.03 * k * k if small else 0.0)], -1)
    p = nominal + _u(g, (E, N, 3), -jitter, jitter) * _t([1.0, 1.0, 0.5])
    q = _quat(torch.cat([_u(g, (E, N, 2), -0.05, 0.05), _u(g, (E, 1, 1), -yaw, yaw) + _u(g, (E, N, 1), -yaw, yaw)], -1))
    S = dict(p=p, q=q, v=_u(g, (E, 1, 3), -0.3, 0.3) + _u(g, (E, N, 3), -0.03, 0.03), w=_u(g, (E, N, 3), -0.1, 0.1),
             ip=torch.zeros(E, N, 3, device=DEV, dtype=torch.float64),
             ia=torch.zeros(E, N, 3, device=DEV, dtype=torch.float64),
             a=torch.zeros(E, N, 4, device=DEV, dtype=torch.float64))
    return {n: x.float().double() for n, x in S.items()}, nominal


def _planes(S):
    """The library's [6, n, 4] float32 state planes of a state of [E, N, .] (or [n, .]) arrays."""
    f = {n: x.reshape(-1, x.shape[-1]) for n, x in S.items()}
    z = torch.zeros_like(f["p"][:, :1])
    return torch.stack([torch.cat([f["p"], f["q"][:, :1]], 1), torch.cat([f["q"][:, 1:], f["v"][:, :1]], 1),
                        torch.cat([f["v"][:, 1:], f["w"][:, :2]], 1), torch.cat([f["w"][:, 2:], f["ip"]], 1),
                        torch.cat([f["ia"], z], 1), f["a"]])


def _actions(kind, E, N, nominal, g, steps, spread=0.1):
    """[steps, E, N, 4] actions of one type (waypoints are the same every step)."""
    if kind == "pid":
        shift = torch.cat([_u(g, (E, 1, 2), -1, 1), _u(g, (E, 1, 1), -0.1, 0.3)], -1)
        yaw = _u(g, (E, 1, 1), -0.5, 0.5).expand(E, N, 1)
        wp = torch.cat([nominal + shift + _u(g, (E, N, 3), -0.02, 0.02), yaw], -1).float().double()
        return wp.expand(steps, E, N, 4)
    if kind == "rpm":
        return (HOVER * _u(g, (steps, E, N, 4), 1 - spread, 1 + spread)).float().double()
    u = _u(g, (steps, E, N, 4), -1, 1)
    if kind == "vel":
        return u * torch.tensor([0.5, 0.5, 0.5, 1.0], device=DEV, dtype=torch.float64)
    scale = torch.tensor([0.1 * MASS * G0, 0.2, 0.2, 1.0], device=DEV, dtype=torch.float64)
    return (u * scale + torch.tensor([MASS * G0, 0, 0, 0], device=DEV, dtype=torch.float64)).float().double()


ACT = dict(rpm=mdg.ACT_RPM, pid=mdg.ACT_PID, vel=mdg.ACT_VEL, attitude=mdg.ACT_ATTITUDE, mixed=mdg.ACT_MIXED)


def _groups(case, seed):
    """The case's swarm as groups of environments of one size: a list of dicts with the environments'
    indices, their first drones, the state [E, N, .], the actions [K, E, N, 4], physics flags [E] and
    a mask of the environments that take waypoints; and the drones of each environment."""
    g = _gen(seed)
    steps = case.get("steps", 1)
    if case["drones"]:
        E, N = case["envs"], case["drones"]
        S, nominal = _formation(E, N, g)
        act = _actions(case["action"], E, N, nominal, g, steps, 0.1 if steps <= 8 else 0.02)
        if case["kind"] == "surrogate":
            S["p"][:: 512, :, 2] += 40.0  # far outside what the network was trained on
        return [dict(env=torch.arange(E, device=DEV), first=torch.arange(E, device=DEV) * N, S=S, act=act,
                     flags=torch.full((E,), 7, device=DEV), pid=None)], np.full(E, N, np.int32)
    E = case["envs"]
    # every size equally often, so that the drone count is the same for every seed
    sizes = np.resize(np.asarray(UNEVEN_SIZES, np.int32), E)[torch.randperm(E, generator=g, device=DEV).cpu()]
    flags = torch.randint(8, (E,), generator=g, device=DEV)
    pid = torch.rand(E, generator=g, device=DEV) < 0.5
    first = torch.as_tensor(np.concatenate([[0], np.cumsum(sizes)[:-1]]), device=DEV)
    out = []
    for N in sorted(set(sizes.tolist())):
        env = torch.as_tensor(np.nonzero(sizes == N)[0], device=DEV)
        S, nominal = _formation(len(env), N, g)
        rpm = _actions("rpm", len(env), N, nominal, g, steps, 0.02)
        wp = _actions("pid", len(env), N, nominal, g, steps)
        out.append(dict(env=env, first=first[env], S=S, act=torch.where(pid[env][:, None, None], wp, rpm),
                        flags=flags[env], pid=pid[env]))
    return out, sizes


def _rows(grp):
    """The global drone indices of a group's drones, in its own order."""
    N = grp["S"]["p"].shape[1]
    return (grp["first"][:, None] + torch.arange(N, device=DEV)).reshape(-1)


def _constants(case):
    c = mdg.Constants.cf2x()
    if case.get("integrator") == "rk4":
        c.integrator = mdg.INTEGRATOR_RK4
    return c


def _swarm(case, seed):
    """(handle, initial state planes, actions [K, n, 4], action type) of a case's swarm."""
    grps, sizes = _groups(case, seed)
    n, K = int(sizes.sum()), case.get("steps", 1)
    planes = torch.zeros(6, n, 4, device=DEV)
    act = torch.zeros(K, n, 4, device=DEV)
    flags = np.zeros(len(sizes), np.uint32)
    types = np.zeros(len(sizes), np.uint8)
    for grp in grps:
        r = _rows(grp)
        planes[:, r] = _planes(grp["S"]).float()
        act[:, r] = grp["act"].reshape(K, -1, 4).float()
        flags[grp["env"].cpu()] = grp["flags"].cpu().numpy()
        if grp["pid"] is not None:
            types[grp["env"].cpu()] = grp["pid"].cpu().numpy()
    h = mdg.Handle(sizes, flags, _constants(case))
    if case["action"] == "mixed":
        h.set_action_types(types)
    return h, planes, act, ACT[case["action"]]


def _mlp_rows(rows, g):
    """Standardised network inputs [rows, 64] in bf16 (41 used)."""
    x = torch.zeros(rows, 64, device=DEV)
    x[:, :41] = torch.randn(rows, 41, generator=g, device=DEV)
    return x.bfloat16()


def _init(seed):
    """Initial network parameters, flat, with small biases."""
    layers = wl.mlp_init(int(seed) % 1000)
    r = np.random.RandomState(int(seed) % (1 << 31))
    return mdg.mlp_flatten([(W, r.uniform(-0.05, 0.05, b.shape).astype(np.float32)) for W, b in layers])


def _normalization(S, N):
    """Statistics of the surrogate's inputs and outputs that the formations stay within."""
    hover = np.full(4, HOVER)
    z = S["p"][..., 2].reshape(-1)
    zc, zs = float(z[z < 20].mean()), 0.5 * float(z[z < 20].max() - z[z < 20].min()) + 0.5
    mean = np.concatenate([[0, 0, zc], [1, 0, 0, 0], np.zeros(6), hover, np.zeros(24)])
    std = np.concatenate([[1.5, 1.5, zs], [0.1, 0.1, 0.1, 0.1], [0.2] * 3, [0.3] * 3, [0.6 * HOVER] * 4,
                          [2.0, 2.0, 2.5, 0.4, 0.4, 0.4] * 4])
    return [a.astype(np.float32) for a in (mean, std, np.zeros(13),
                                           np.array([0.01] * 3 + [0.005] * 4 + [0.1] * 3 + [0.3] * 3),
                                           mean - 4 * std, mean + 4 * std)]


def _transitions(rows, g):
    """A transition set of the shape a swarm gives: columns of different centres and scales, a heavy
    tail from near-coincident heights in the changes, and a few non-finite rows."""
    raw = torch.randn(rows, 41, generator=g, device=DEV)
    raw *= _u(g, (41,), 0.05, 3.0).float()
    raw += _u(g, (41,), -2.0, 2.0).float()
    raw[:, 13:17] = raw[:, 13:17] * 200 + HOVER
    raw[:, 35:41] = 0.0  # environments of four drones have three neighbours
    delta = torch.randn(rows, 13, generator=g, device=DEV) * _u(g, (13,), 0.01, 0.5).float()
    tail = torch.rand(rows, generator=g, device=DEV) < 0.02
    delta[tail, 7:10] *= 1.0 / (torch.rand(int(tail.sum()), 3, generator=g, device=DEV) ** 2 + 1e-3)
    delta[torch.randint(rows, (max(1, rows // 100000),), generator=g, device=DEV), 2] = float("nan")
    return raw, delta


def _wanted(case, obs):
    """KIN, neighbours and, in swarms of up to eight drones, their relative states. (Among more drones
    two neighbours at distances that round alike swap places, and their relative states with them.)"""
    return obs if 0 < case["drones"] <= 8 else obs[:2]


# ---------------------------------------------------------------- preparing and running
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=dict(case))
    if kind == "step":
        h, init, act, code = _swarm(case, seed)
        s.update(h=h, init=init, act=act, code=code, state=init.clone(), obs=_wanted(case, h.new_obs()), restore=[])
        s["restore"].append((s["state"], s["init"]))
        if case["randomize"]:
            table = torch.as_tensor(wl.dr_table(int(seed) % 1000, case["envs"], depth=3), device=DEV)
            live = h.new_randomization_state(3)
            h.set_randomization(table, *live, seed=int(seed) % 1000)
            s.update(table=table, live=live)
            s["restore"] += [(x, x.clone()) for x in live]
        if case["graph"]:
            _steps(s)
            torch.cuda.synchronize()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                _steps(s)
    elif kind == "rollout":
        h, init, act, code = _swarm(case, seed)
        K, n = case["steps"], h.n
        if case["action"] == "pid":
            act = act[0].contiguous()
        lead = (K,) if case["every"] else ()
        obs = (torch.empty(lead + (n, 20), device=DEV), torch.empty(lead + (n, 4), dtype=torch.int32, device=DEV),
               torch.empty(lead + (n, 24), device=DEV))
        s.update(h=h, init=init, act=act, code=code, state=init.clone(), obs=_wanted(case, obs),
                 mode=mdg.OBS_EVERY_STEP if case["every"] else mdg.OBS_LAST)
    elif kind == "render":
        g = _gen(seed)
        S, _ = _formation(case["envs"], case["drones"], g, yaw=math.pi)
        h = mdg.Handle(np.full(case["envs"], case["drones"], np.int32), np.full(case["envs"], 7, np.uint32))
        s.update(h=h, state=_planes(S).float(), frames=h.new_frames(depth=False))
    elif kind == "network":
        g = _gen(seed)
        x = _mlp_rows(case["rows"], g)
        s.update(mlp=mdg.MLP(case["rows"], _init(seed)), x=x, y=torch.empty(case["rows"], 32, device=DEV))
    elif kind == "surrogate":
        grps, sizes = _groups(case, seed)
        h, init, act, code = _swarm(case, seed)
        mlp = mdg.MLP((h.n + 127) // 128 * 128, _init(seed))
        mlp.set_normalization(*_normalization(grps[0]["S"], case["drones"]))
        s.update(h=h, init=init, state=init.clone(), act=act[0].contiguous(), code=code, mlp=mlp,
                 fallbacks=torch.zeros(1, dtype=torch.int32, device=DEV))
    elif kind == "train":
        x, t, _ = _training(case, seed)
        s.update(mlp=mdg.MLP(case["batch"], _init(seed)), x=x, t=t, loss=torch.zeros(case["batches"], 1, device=DEV))
    elif kind == "transition":
        h, init, act, _ = _swarm(dict(case, action="rpm"), seed)
        n = h.n
        g = _gen(int(seed) + 1)
        s.update(h=h, init=init, state=init.clone(), rpm=act[0].contiguous(), scale=_u(g, (n, 4), 0.98, 1.02).float(),
                 applied=torch.empty(n, 4, device=DEV), raw=torch.empty(n, 41, device=DEV),
                 delta=torch.empty(n, 13, device=DEV))
    else:
        raw, delta = _transitions(case["rows"], _gen(seed))
        s.update(mlp=mdg.MLP(128), raw=raw, delta=delta,
                 x=torch.zeros(case["rows"], 64, dtype=torch.bfloat16, device=DEV),
                 t=torch.zeros(case["rows"], 32, device=DEV))
    return s


def _training(case, seed):
    g = _gen(seed)
    x = torch.stack([_mlp_rows(case["batch"], g) for _ in range(case["batches"])])
    A = torch.randn(41, 13, generator=g, device=DEV) / math.sqrt(41)
    t = torch.zeros(case["batches"], case["batch"], 32, device=DEV)
    t[..., :13] = torch.tanh(x[..., :41].float() @ A) + 0.1 * torch.randn(
        case["batches"], case["batch"], 13, generator=g, device=DEV)
    return x, t, 1e-3


def _steps(s):
    """An episode's start (the buffers restored) and its control steps."""
    for live, start in s["restore"]:
        live.copy_(start)
    for k in range(s["case"]["steps"]):
        s["h"].step_obs(s["state"], s["act"][k], s["code"], SUBSTEPS, *s["obs"])


def _outputs(state, kin=None, idx=None, rel=None):
    """Outputs in whole, the motor speeds (thousands) apart from the quantities of order one."""
    out = dict(state=state[:5], speeds=state[5])
    if kin is not None:
        out.update(kin=kin[..., :16], kin_speeds=kin[..., 16:], idx=idx)
    if rel is not None:
        out.update(rel=rel)
    return out


def run(s):
    kind = s["case"]["kind"]
    if kind == "step":
        if "graph" in s:
            s["graph"].replay()
        else:
            _steps(s)
        out = _outputs(s["state"], *s["obs"])
        if "live" in s:
            out.update(motor=s["live"][0], wind=s["live"][2])
        return out
    if kind == "rollout":
        s["state"].copy_(s["init"])
        s["h"].rollout(s["state"], s["act"], s["code"], SUBSTEPS, s["case"]["steps"], s["mode"], *s["obs"])
        return _outputs(s["state"], *s["obs"])
    if kind == "render":
        s["h"].render(s["state"], *s["frames"])
        return dict(rgba=s["frames"][0], seg=s["frames"][2])
    if kind == "network":
        s["mlp"].forward(s["x"], s["y"])
        return s["y"]
    if kind == "surrogate":
        s["state"].copy_(s["init"])
        s["mlp"].step(s["h"], s["state"], s["act"], s["code"], SUBSTEPS, 4.0, s["fallbacks"])
        return dict(_outputs(s["state"]), fallbacks=s["fallbacks"])
    if kind == "train":
        for x, t, loss in zip(s["x"], s["t"], s["loss"]):
            s["mlp"].grad(x, t, loss)
            s["mlp"].adam(1e-3)
        return dict(loss=s["loss"], grads=s["mlp"].grads(), params=s["mlp"].params())
    if kind == "transition":
        s["state"].copy_(s["init"])
        s["h"].transition(s["state"], s["rpm"], s["applied"], s["raw"], s["delta"], s["scale"], SUBSTEPS)
        return dict(_outputs(s["state"]), applied=s["applied"], raw=s["raw"], delta=s["delta"])
    finite, kept = s["mlp"].fit_normalization(s["raw"], s["delta"], s["x"], s["t"])
    # the whole buffers: the rows beyond `kept` stay zero
    return dict(x=s["x"], t=s["t"], finite=finite, kept=kept, norm=list(s["mlp"].normalization()))


# ---------------------------------------------------------------- work and tolerances
def _drones(case):
    """(drones, ordered pairs of drones of one environment) of a case, on average for uneven swarms."""
    sizes = UNEVEN_SIZES if not case["drones"] else (case["drones"],)
    n = case["envs"] * sum(sizes) / len(sizes)
    return n, case["envs"] * sum(N * (N - 1) for N in sizes) / len(sizes)


def work(case):
    kind = case["kind"]
    if kind in ("network", "train"):
        macs = 41 * 256 + 2 * 256 * 256 + 256 * 13
        rows = case["rows"] if kind == "network" else case["batch"] * case["batches"]
        if kind == "network":
            return dict(bytes=rows * (128 + 128) + 2 * 156448, flops=2 * macs * rows)
        # the first layer's input gradient is not needed
        return dict(bytes=rows * (128 + 128) + 4 * 156448 * 7 * case["batches"],
                    flops=2 * rows * (3 * macs - 41 * 256))
    if kind == "dataset":
        return dict(bytes=case["rows"] * (54 * 4 + 128 + 128), flops=case["rows"] * 54 * 8)
    n, pairs = _drones(case)
    # per substep: motor to exponential map ~170 operations, 23 a downwash pair; Runge-Kutta takes four
    # evaluations and 100 operations of combination; the controller ~150, an observation ~80 and 10 a pair
    euler = n * 170 + pairs * 23
    sub = (4 * euler + n * 100) if case.get("integrator") == "rk4" else euler
    obs = n * (80 + 16 + (96 if 0 < case["drones"] <= 8 else 0))
    obs_ops = n * 80 + pairs * 10
    steps = case.get("steps", 1)
    if kind == "step":
        # per step: state and action read, state and observations written
        b, f = n * (80 + 16 + 96) + obs, SUBSTEPS * sub + n * 150 + obs_ops
        if case["randomize"]:  # rotor speeds and the action history both ways, a row and the wind per environment
            b += n * (32 + 96) + case["envs"] * (160 + 64)
            f += n * 600
        return dict(bytes=steps * b, flops=steps * f)
    if kind == "rollout":
        k_obs = steps if case["every"] else 1
        return dict(bytes=n * (80 + 96) + n * 16 * (1 if case["action"] == "pid" else steps) + k_obs * obs,
                    flops=steps * (SUBSTEPS * sub + n * 150) + k_obs * obs_ops)
    if kind == "render":
        return dict(bytes=n * (48 * 64 * 8 + 32), flops=n * 48 * 64 * 30)
    if kind == "surrogate":
        return dict(bytes=n * (80 + 16 + 96), flops=n * 2 * (41 * 256 + 2 * 256 * 256 + 256 * 13) + obs_ops + n * 150)
    return dict(bytes=n * (80 + 32 + 96 + 16 + 164 + 52), flops=SUBSTEPS * sub + obs_ops)


def tolerance(case):
    """About four times the largest difference from `exact` that was measured over listed and drawn cases."""
    kind = case["kind"]
    if kind == "network":  # bf16 weights and activations: 4.5e-3, at most 4e-2
        return dict(rel=2e-2, max=0.16)
    if kind == "train":  # gradients 7e-3, at most 0.17; loss 5e-4; parameters 7e-4
        return dict(rel=3e-2, max=0.6)
    if kind == "surrogate":  # the network's error on the state change: 1.4e-4, at most 2.3e-3
        return dict(rel=5e-4, max=1e-2, differ=1e-4)
    if kind == "dataset":  # inputs in bf16: 1.7e-3, at most 3.9e-3; targets 5e-8
        return dict(rel=7e-3, max=1.6e-2, differ=1e-4)
    if kind == "render":  # a channel rounds to the other side: 1.4e-4; segmentation 1e-7
        return dict(differ=6e-4)
    # single precision over up to 160 substeps: 2.4e-6, at most 1.4e-3 where a wake amplifies it; neighbours 2e-5
    return dict(rel=1e-5, max=6e-3, differ=1e-4)


# ---------------------------------------------------------------- the paths in float64
MASS, ARM, G0, KF, KM, RP = 0.027, 0.0397, 9.81, 3.16e-10, 7.94e-12, 0.02325
INERTIA = (1.4e-5, 1.4e-5, 2.17e-5)
DT, DT_CTRL = 1 / 240, 1 / 48
C_GND, C_XY, C_Z = 11.36859, 9.1785e-7, 10.311e-7
H_CLIP = 0.25 * RP * math.sqrt(C_GND / 1.25)
HOVER, MAX_RPM = math.sqrt(MASS * G0 / (4 * KF)), math.sqrt(2.25 * MASS * G0 / (4 * KF))
POS_GAINS = ((0.4, 0.4, 1.0), (0.01, 0.01, 0.01), (0.9, 0.9, 2.0))
ATT_GAINS = ((2e-3, 2e-3, 1e-3), (0.0, 0.0, 1e-4), (5e-4, 5e-4, 2e-4))
MODEL = dict(mass=MASS, arm=ARM, g=G0, kf=KF, km=KM, J=INERTIA, cxy=C_XY, cz=C_Z, cgnd=C_GND, c1=2267.18)


def _t(v):
    return torch.tensor(v, device=DEV, dtype=torch.float64)


def _rpy(q):
    w, x, y, z = q.unbind(-1)
    return torch.stack([torch.atan2(2 * (w * x + y * z), 1 - 2 * (x * x + y * y)),
                        torch.asin((2 * (w * y - z * x)).clamp(-1, 1)),
                        torch.atan2(2 * (w * z + x * y), 1 - 2 * (y * y + z * z))], -1)


def _rotation(q):
    w, x, y, z = q.unbind(-1)
    rows = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(rows, -1).reshape(q.shape[:-1] + (3, 3))


def _control(S, act, kind):
    """Action -> RPMs with the cascaded controller; updates the integrals of S."""
    if kind == "rpm":
        return act.clamp(0, MAX_RPM)
    kp, ki, kd = (_t(x) for x in POS_GAINS)
    akp, aki, akd = (_t(x) for x in ATT_GAINS)
    rpy = _rpy(S["q"])
    e_rate = torch.zeros_like(S["w"])
    if kind == "attitude":
        T, tilt, yaw_t, e_rate[..., 2] = act[..., 0], act[..., 1:3], rpy[..., 2], act[..., 3]
    else:
        if kind == "pid":
            e = act[..., :3] - S["p"]
            S["ip"] = (S["ip"] + e * DT_CTRL).clamp(-2, 2)
            acc = kp * e + ki * S["ip"] - kd * S["v"]
            yaw_t = act[..., 3]
        else:
            vt = torch.einsum("...ij,...j->...i", _rotation(S["q"]), act[..., :3])
            S["ip"] = S["ip"].clamp(-2, 2)
            acc = ki * S["ip"] + kd * (vt - S["v"])
            yaw_t, e_rate[..., 2] = rpy[..., 2], act[..., 3]
        acc = acc + _t([0, 0, G0])
        T = MASS * acc.norm(dim=-1)
        s, c = torch.sin(yaw_t), torch.cos(yaw_t)
        tilt = torch.stack([acc[..., 0] * s - acc[..., 1] * c, acc[..., 0] * c + acc[..., 1] * s], -1) / G0
    e = torch.cat([tilt, yaw_t[..., None]], -1) - rpy
    e = torch.cat([e[..., :2], torch.remainder(e[..., 2:] + math.pi, 2 * math.pi) - math.pi], -1)
    S["ia"] = (S["ia"] + e * DT_CTRL).clamp(-0.5, 0.5)
    tau = akp * e + aki * S["ia"] + akd * (e_rate - S["w"])
    tx, ty, tz = (tau * _t([math.sqrt(2) / ARM, math.sqrt(2) / ARM, KF / KM])).unbind(-1)
    f = 0.25 * torch.stack([T + tx - ty - tz, T + tx + ty + tz, T - tx + ty - tz, T - tx - ty + tz], -1)
    return torch.sqrt(f.clamp(0, KF * MAX_RPM ** 2) / KF)


def _forces(S, rpm, flags, c, extra=0.0):
    """World force and body angular acceleration of drones [E, N] (flags [E])."""
    n2 = rpm * rpm
    F = (c["kf"][..., None] if torch.is_tensor(c["kf"]) else c["kf"]) * n2
    T = F.sum(-1)
    l = c["arm"] / math.sqrt(2)
    tau = torch.stack([l * (F[..., 0] + F[..., 1] - F[..., 2] - F[..., 3]),
                       l * (F[..., 1] + F[..., 2] - F[..., 0] - F[..., 3]),
                       c["km"] * (n2[..., 1] + n2[..., 3] - n2[..., 0] - n2[..., 2])], -1)
    R = _rotation(S["q"])
    up = R[..., :, 2]
    f = up * T[..., None]
    fz = -c["mass"] * c["g"] + torch.zeros_like(T)
    gnd, drag, dw = (((flags & b) != 0)[:, None] for b in (GND, DRAG, DW))
    h = S["p"][..., 2].clamp(min=H_CLIP)
    ok = gnd & (R[..., 2, 2] > 0) & (R[..., 2, 0].abs() < 1)
    fz = fz + torch.where(ok, c["cgnd"] * (RP / 4) ** 2 * T / (h * h), 0.0)
    k = 2 * math.pi / 60 * rpm.sum(-1)
    rv = (up * S["v"]).sum(-1)
    d = (k * c["cxy"])[..., None] * S["v"] + (k * (c["cz"] - c["cxy"]) * rv)[..., None] * up
    f = f - torch.where(drag[..., None], d, 0.0)
    p = S["p"]
    dz = p[:, None, :, 2] - p[:, :, None, 2]
    d2 = (p[:, None, :, :2] - p[:, :, None, :2]).square().sum(-1)
    beta2 = (0.16 * dz - 0.11).square().clamp(min=1e-12)
    up_of = (dz > 0) & (d2 < 100.0)
    c1 = c["c1"].unsqueeze(-1) if torch.is_tensor(c["c1"]) else c["c1"]
    wake = c1 * (RP / 4) ** 2 / dz.square() * torch.exp(-0.5 * d2 / beta2)
    fz = fz - torch.where(dw, torch.where(up_of, wake, 0.0).sum(-1), 0.0)
    f = torch.cat([f[..., :2], f[..., 2:] + fz[..., None]], -1) + extra
    J = c["J"] if torch.is_tensor(c["J"]) else _t(c["J"])
    return f, (tau - torch.linalg.cross(S["w"], J * S["w"])) / J


def _qmul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _mass(c):
    return c["mass"][..., None] if torch.is_tensor(c["mass"]) else c["mass"]


def _euler(S, rpm, flags, c=MODEL, extra=0.0):
    f, wd = _forces(S, rpm, flags, c, extra)
    nw = S["w"].norm(dim=-1, keepdim=True)
    th = 0.5 * DT * nw
    k = torch.where(nw > 0, torch.sin(th) / nw.clamp(min=1e-300), 0.5 * DT)
    q = _qmul(S["q"], torch.cat([torch.cos(th), k * S["w"]], -1))
    return dict(S, p=S["p"] + DT * S["v"], q=q / q.norm(dim=-1, keepdim=True), v=S["v"] + DT * f / _mass(c),
                w=S["w"] + DT * wd)


def _rk4(S, rpm, flags, c=MODEL):
    def rate(x):
        unit = dict(x, q=x["q"] / x["q"].norm(dim=-1, keepdim=True))
        f, wd = _forces(unit, rpm, flags, c)
        w0 = torch.cat([torch.zeros_like(x["w"][..., :1]), x["w"]], -1)
        return dict(p=x["v"], q=0.5 * _qmul(x["q"], w0), v=f / c["mass"], w=wd)

    def at(k, hstep):
        return dict(S, **{n: S[n] + hstep * k[n] for n in k})
    k1 = rate(S)
    k2 = rate(at(k1, DT / 2))
    k3 = rate(at(k2, DT / 2))
    k4 = rate(at(k3, DT))
    out = at({n: k1[n] + 2 * k2[n] + 2 * k3[n] + k4[n] for n in k1}, DT / 6)
    return dict(out, q=out["q"] / out["q"].norm(dim=-1, keepdim=True))


def _neighbours(S):
    """(local indices [E, N, 4], -1 where fewer, relative states [E, N, 24])."""
    p = S["p"]
    E, N = p.shape[:2]
    d2 = (p[:, None] - p[:, :, None]).square().sum(-1)
    d2 = d2 + torch.diag(torch.full((N,), float("inf"), device=DEV, dtype=torch.float64))
    m = min(4, N - 1)
    idx = torch.sort(d2, dim=-1, stable=True).indices[..., :m]
    pv = torch.cat([S["p"], S["v"]], -1)
    rel = torch.zeros(E, N, 4, 6, device=DEV, dtype=torch.float64)
    if m:
        rel[:, :, :m] = torch.gather(pv[:, None].expand(E, N, N, 6), 2,
                                     idx[..., None].expand(E, N, m, 6)) - pv[:, :, None]
    full = torch.full((E, N, 4), -1, device=DEV, dtype=torch.int64)
    full[..., :m] = idx
    return full, rel.reshape(E, N, 24)


def _observe(S, first):
    idx, rel = _neighbours(S)
    kin = torch.cat([S["p"], S["q"], _rpy(S["q"]), S["v"], S["w"], S["a"]], -1)
    idx = torch.where(idx >= 0, idx + first[:, None, None], idx).int()
    return [x.reshape(-1, x.shape[-1]) for x in (kin, idx, rel)]


def _step(S, act, kind, flags, pid=None, rk4=False):
    if pid is None:
        rpm = _control(S, act, kind)
    else:
        held = dict(S)
        wp = _control(S, act, "pid")
        m = pid[:, None, None]
        for n in ("ip", "ia"):
            S[n] = torch.where(m, S[n], held[n])
        rpm = torch.where(m, wp, _control(S, act, "rpm"))
    for _ in range(SUBSTEPS):
        S = (_rk4 if rk4 else _euler)(S, rpm, flags)
    return dict(S, a=rpm)


# -- counter-based draws: SplitMix64 over (seed, stream, step, index, component)
def _wrap(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _mix(z):
    def shift(x, k):
        return (x >> k) & ((1 << (64 - k)) - 1)
    z = z + _wrap(0x9E3779B97F4A7C15)
    z = (z ^ shift(z, 30)) * _wrap(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * _wrap(0x94D049BB133111EB)
    return z ^ shift(z, 31)


def _uniform(seed, stream, step, index, comp):
    h = _mix(torch.full_like(index, int(seed)))
    h = _mix(_mix(_mix(_mix(h ^ stream) ^ step) ^ index) ^ comp)
    return ((h >> 40) & 0xFFFFFF).double() / (1 << 24)


def _gauss(seed, stream, step, index, m):
    """The two normals of Box and Muller's transform of components 2m and 2m + 1."""
    r = torch.sqrt(-2 * torch.log(1 - _uniform(seed, stream, step, index, 2 * m)))
    a = 2 * math.pi * _uniform(seed, stream, step, index, 2 * m + 1)
    return r * torch.cos(a), r * torch.sin(a)


def _noisy(kin, row, seed, step, drone):
    xi = torch.stack([x for m in range(6) for x in _gauss(seed, 22, step, drone, m)], -1)
    sigma = torch.stack([row[:, k] for k in (32, 34, 33, 35)], -1)[:, None]  # p, rpy, v, w
    noise = xi * sigma.repeat_interleave(3, -1)
    return torch.cat([kin[..., :3] + noise[..., :3], kin[..., 3:7], kin[..., 7:10] + noise[..., 3:6],
                      kin[..., 10:13] + noise[..., 6:9], kin[..., 13:16] + noise[..., 9:12], kin[..., 16:]], -1)


def _randomized(case, seed):
    grp = _groups(case, seed)[0][0]
    S, first, flags = grp["S"], grp["first"], grp["flags"]
    E, N = S["p"].shape[:2]
    key = int(seed) % 1000
    row = torch.as_tensor(wl.dr_table(key, E, depth=3), device=DEV).double()
    env, drone = grp["env"], _rows(grp).reshape(E, N)
    b = {k: row[:, k, None] for k in range(36)}
    c = dict(mass=MASS * b[0], arm=ARM * b[4], g=G0 * b[16], kf=KF * b[5], km=KM * b[6],
             J=_t(INERTIA) * row[:, None, 1:4], cxy=C_XY * b[7], cz=C_Z * b[8], cgnd=C_GND * b[9], c1=2267.18 * b[10])
    hist, motor, kin = None, None, None
    dry = torch.zeros(E, 3, device=DEV, dtype=torch.float64)
    phase = torch.full((E,), -1.0, device=DEV)
    gust = torch.zeros(E, 3, device=DEV, dtype=torch.float64)
    delay, late = row[:, 18].long()[:, None, None, None], (row[:, 36] == 1)[:, None, None]
    for k in range(case["steps"]):
        got = grp["act"][k]
        hist = torch.stack([got, got, got], 2) if hist is None else torch.cat([got[:, :, None], hist[:, :, :2]], 2)
        act = torch.gather(hist, 2, delay.expand(E, N, 1, 4))[:, :, 0]
        before = _noisy(torch.cat([S["p"], S["q"], _rpy(S["q"]), S["v"], S["w"], S["a"]], -1), row, key, k, drone)
        rpm = _control(S, act, case["action"])
        L = row[:, 31] / (0.177 + 8.23e-4 * row[:, 31]) ** 1.2
        alpha = torch.exp(-DT_CTRL * row[:, 28] / L)
        (x0, y0), (z0, _) = _gauss(key, 21, k, env, 0), _gauss(key, 21, k, env, 1)
        sc = row[:, 27] * torch.sqrt((1 - alpha * alpha).clamp(min=0))
        dry = alpha[:, None] * dry + sc[:, None] * torch.stack([x0, y0, z0], -1)
        start = (phase < 0) & (_uniform(key, 21, k, env, 4) < row[:, 24])
        gz, ang = 2 * _uniform(key, 21, k, env, 5) - 1, 2 * math.pi * _uniform(key, 21, k, env, 6)
        rho = torch.sqrt((1 - gz * gz).clamp(min=0))
        gust = torch.where(start[:, None], torch.stack([rho * torch.cos(ang), rho * torch.sin(ang), gz], -1), gust)
        phase = torch.where(start, torch.zeros_like(phase), phase)
        on = phase >= 0
        amp = torch.where(on, row[:, 25] * torch.sin(math.pi * phase.double()), 0.0)
        nxt = phase + torch.tensor(DT_CTRL, dtype=torch.float32, device=DEV) / row[:, 26].float()
        phase = torch.where(on, torch.where(nxt > 1, torch.full_like(nxt, -1.0), nxt), phase)
        wt = row[:, 30] * (k * DT_CTRL)
        force = amp[:, None] * gust + row[:, 29, None] * torch.stack(
            [torch.sin(wt), torch.cos(wt), 0.3 * torch.sin(2 * wt)], -1)
        vr = (row[:, 20:23] + dry)[:, None] - S["v"]
        extra = force[:, None] + b[23][..., None] * vr.norm(dim=-1, keepdim=True) * vr
        cmd = torch.minimum(rpm * row[:, None, 12:16], MAX_RPM * b[11][..., None])
        motor = cmd if motor is None else motor
        lag = torch.exp(-DT / b[17][..., None])
        for _ in range(SUBSTEPS):
            motor = cmd + (motor - cmd) * lag
            S = _euler(S, motor, flags, c, extra)
        S = dict(S, a=rpm)
        after = _noisy(torch.cat([S["p"], S["q"], _rpy(S["q"]), S["v"], S["w"], S["a"]], -1), row, key, k, drone)
        kin = torch.where(late, before, after)
    _, idx, rel = _observe(S, first)
    wind = torch.cat([dry, phase[:, None].double(), gust,
                      torch.full((E, 1), float(case["steps"]), device=DEV, dtype=torch.float64)], -1)
    return dict(_outputs(_planes(S), *_wanted(case, (kin.reshape(-1, 20), idx, rel))), motor=motor.reshape(-1, 4),
                wind=wind)


def _flight(case, seed):
    grps, sizes = _groups(case, seed)
    n, K = int(sizes.sum()), case["steps"]
    every = case.get("every", False)
    lead = (K,) if every else ()
    out = dict(state=torch.zeros(6, n, 4, device=DEV, dtype=torch.float64),
               kin=torch.zeros(lead + (n, 20), device=DEV, dtype=torch.float64),
               idx=torch.zeros(lead + (n, 4), device=DEV, dtype=torch.int32),
               rel=torch.zeros(lead + (n, 24), device=DEV, dtype=torch.float64))
    for grp in grps:
        S, r = grp["S"], _rows(grp)
        for k in range(K):
            S = _step(S, grp["act"][k], case["action"], grp["flags"], grp["pid"], case.get("integrator") == "rk4")
            if every or k == K - 1:
                for name, x in zip(("kin", "idx", "rel"), _observe(S, grp["first"])):
                    (out[name][k] if every else out[name])[r] = x
        out["state"][:, r] = _planes(S)
    return _outputs(out["state"], *_wanted(case, (out["kin"], out["idx"], out["rel"])))


def _network(flat, x):
    """The network on float64 inputs [rows, 64] (rows in chunks)."""
    layers = [(_t(W), _t(b)) for W, b in mdg.mlp_unflatten(np.asarray(flat, np.float64))]
    y = []
    for part in x.split(32768):
        h = part.double()
        for i, (W, b) in enumerate(layers):
            h = h @ W.T + b
            h = h * torch.sigmoid(h) if i < 3 else h
        y.append(h)
    return torch.cat(y)


def _features(S, rpm):
    x = torch.cat([S["p"], S["q"], S["v"], S["w"], rpm, _neighbours(S)[1]], -1)
    return x.reshape(-1, 41)


def _surrogate(case, seed):
    grp = _groups(case, seed)[0][0]
    S, flags = dict(grp["S"]), grp["flags"]
    E, N = S["p"].shape[:2]
    mean, std, out_mean, out_std, lo, hi = (_t(a.astype(np.float64)) for a in _normalization(grp["S"], N))
    rpm = _control(S, grp["act"][0], case["action"])
    raw = _features(S, rpm)
    z = (raw - mean) / std
    far = ((z.abs() > 4.0) | (raw < lo) | (raw > hi)).any(-1).reshape(E, N).any(-1)
    x = torch.zeros(E * N, 64, device=DEV, dtype=torch.float64)
    x[:, :41] = z
    d = (out_mean + out_std * _network(_init(seed), x)[:, :13]).reshape(E, N, 13)
    q = S["q"] + d[..., 3:7]
    net = dict(S, p=S["p"] + d[..., :3], q=q / q.norm(dim=-1, keepdim=True), v=S["v"] + d[..., 7:10],
               w=S["w"] + d[..., 10:13])
    plain = S
    for _ in range(SUBSTEPS):
        plain = _euler(plain, rpm, flags)
    out = {k: torch.where(far[:, None, None], plain[k], net[k]) for k in S}
    return dict(_outputs(_planes(dict(out, a=rpm))), fallbacks=far.sum()[None].int())


def _train(case, seed):
    x, t, lr = _training(case, seed)
    P = [_t(a.astype(np.float64)).requires_grad_() for W, b in mdg.mlp_unflatten(_init(seed)) for a in (W, b)]
    m, v = [torch.zeros_like(p) for p in P], [torch.zeros_like(p) for p in P]
    losses = []
    for k in range(case["batches"]):
        h = x[k].double()
        for i in range(4):
            h = h @ P[2 * i].T + P[2 * i + 1]
            h = h * torch.sigmoid(h) if i < 3 else h
        loss = (h[:, :13] - t[k, :, :13].double()).square().mean()
        grads = torch.autograd.grad(loss, P)
        losses.append(loss.detach())
        with torch.no_grad():
            for j, g in enumerate(grads):
                m[j] = 0.9 * m[j] + 0.1 * g
                v[j] = 0.999 * v[j] + 0.001 * g * g
                P[j] -= lr * (m[j] / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v[j] / (1 - 0.999 ** (k + 1))) + 1e-8)
    flat = [torch.cat([a.detach().reshape(-1) for a in arrs]).cpu().numpy() for arrs in (grads, P)]
    return dict(loss=torch.stack(losses)[:, None], grads=flat[0], params=flat[1])


def _transition(case, seed):
    s = prepare(case, seed)
    grp = _groups(dict(case, action="rpm"), seed)[0][0]
    S = grp["S"]
    applied = (s["rpm"] * s["scale"]).double()
    rpm = applied.reshape(S["a"].shape)
    raw = _features(S, rpm)
    held = rpm.clamp(0, MAX_RPM)
    new = S
    for _ in range(SUBSTEPS):
        new = (_rk4 if case["integrator"] == "rk4" else _euler)(new, held, grp["flags"])
    new = dict(new, a=held)
    x13 = [torch.cat([Z["p"], Z["q"], Z["v"], Z["w"]], -1).reshape(-1, 13) for Z in (S, new)]
    return dict(_outputs(_planes(new)), applied=applied, raw=raw, delta=x13[1] - x13[0])


def _dataset(case, seed):
    raw, delta = _transitions(case["rows"], _gen(seed))
    v = torch.cat([raw, delta], 1).double()
    v = v[torch.isfinite(v).all(1)]
    n_fin = len(v)
    s = torch.sort(v[:: max(1, n_fin // 262144)], dim=0).values
    pos = [(len(s) - 1) * float(np.float32(0.005)), (len(s) - 1) * (1 - float(np.float32(0.005)))]
    lo, hi = (s[int(x)] + (x - int(x)) * (s[min(int(x) + 1, len(s) - 1)] - s[int(x)]) for x in pos)
    box = [(lo - 0.1 * (hi - lo)).float().double(), (hi + 0.1 * (hi - lo)).float().double()]
    v = v[((v >= box[0]) & (v <= box[1])).all(1)]
    mean, sd = v.mean(0), v.std(0)
    sd = torch.where(sd > 1e-6 * mean.abs().clamp(min=1), sd, torch.ones_like(sd))
    z = (v - mean) / sd
    keep = (z[:, :41].abs() <= 4).all(1) & (z[:, 41:].abs() <= 8).all(1)
    z, v = z[keep], v[keep][:, :41]
    a, b = v.min(0).values, v.max(0).values
    pad = 0.1 * (b - a) + 1e-6
    n = len(z) // 128 * 128
    x = torch.zeros(case["rows"], 64, device=DEV, dtype=torch.float64)
    t = torch.zeros(case["rows"], 32, device=DEV, dtype=torch.float64)
    x[:n, :41], t[:n, :13] = z[:n, :41], z[:n, 41:]
    return dict(x=x, t=t, finite=None, kept=None,
                norm=[y.cpu().numpy() for y in (mean[:41], sd[:41], mean[41:], sd[41:], a - pad, b + pad)])


def _camera(case, seed):
    """Frames by ray casting, in chunks of cameras."""
    S, _ = _formation(case["envs"], case["drones"], _gen(seed), yaw=math.pi)
    E, N = S["p"].shape[:2]
    semi = _t([ARM + RP, ARM + RP, 0.3 * (ARM + RP)])
    light = _t([0.3, 0.2, 1.0]) / math.sqrt(0.09 + 0.04 + 1.0)
    th = math.tan(math.pi / 6)
    row, col = torch.meshgrid(torch.arange(48, device=DEV), torch.arange(64, device=DEV), indexing="ij")
    nx = ((col.reshape(-1) + 0.5) / 32 - 1).double() * (th * 64 / 48)
    ny = (1 - (row.reshape(-1) + 0.5) / 24).double() * th
    body = torch.stack([torch.ones_like(nx), -nx, ny], -1)
    palette = _t([[0.90, 0.25, 0.20], [0.20, 0.70, 0.30], [0.20, 0.35, 0.90], [0.95, 0.75, 0.15], [0.70, 0.30, 0.80],
                  [0.15, 0.75, 0.80], [0.95, 0.50, 0.20], [0.60, 0.60, 0.65]])
    R = _rotation(S["q"])
    rgba = torch.empty(E * N, 48 * 64, 4, dtype=torch.uint8, device=DEV)
    seg = torch.empty(E * N, 48 * 64, dtype=torch.int32, device=DEV)
    inf = float("inf")
    for first in range(0, E * N, 1024):
        cam = torch.arange(first, min(first + 1024, E * N), device=DEV)
        e, k = cam // N, cam % N
        o = S["p"][e, k] + 0.02 * R[e, k][:, :, 0]
        d = torch.einsum("cij,xj->cxi", R[e, k], body)
        down = (o[:, None, 2] > 0) & (d[..., 2] < 0)
        best = torch.where(down, -o[:, None, 2] / torch.where(down, d[..., 2], -1.0), inf)
        best = torch.where(best > 1e-4, best, inf)
        g = o[:, None] + torch.where(torch.isfinite(best), best, 0.0)[..., None] * d
        odd = torch.remainder(torch.floor(2 * g[..., 0]) + torch.floor(2 * g[..., 1]), 2) != 0
        hit = torch.isfinite(best)
        color = torch.where(hit[..., None], (torch.where(odd, 0.35, 0.55) * (0.35 + 0.65 * light[2]))[..., None],
                            _t([0.55, 0.70, 0.90]))
        ids = torch.where(hit, 0, -1)
        for j in range(N):
            Rj = R[e, j]
            oj = torch.einsum("cij,ci->cj", Rj, o - S["p"][e, j]) / semi
            dj = torch.einsum("cij,cxi->cxj", Rj, d) / semi
            A, B = dj.square().sum(-1), 2 * (dj * oj[:, None]).sum(-1)
            disc = B * B - 4 * A * (oj.square().sum(-1) - 1)[:, None]
            sq = torch.sqrt(disc.clamp(min=0))
            t1, t2 = (-B - sq) / (2 * A), (-B + sq) / (2 * A)
            tj = torch.where(t1 > 1e-4, t1, torch.where(t2 > 1e-4, t2, inf))
            near = (disc >= 0) & (tj < best) & (k != j)[:, None]
            best = torch.where(near, tj, best)
            nrm = torch.einsum("cij,cxj->cxi", Rj, (oj[:, None] + torch.where(near, tj, 0.0)[..., None] * dj) / semi)
            nl = (nrm * light).sum(-1) / nrm.norm(dim=-1)
            gid = e * N + j
            color = torch.where(near[..., None], palette[gid % 8][:, None] * (0.35 + 0.65 * nl.clamp(min=0))[..., None],
                                color)
            ids = torch.where(near, (gid + 1)[:, None], ids)
        rgba[cam, :, :3] = torch.round(255 * color.clamp(0, 1)).to(torch.uint8)
        seg[cam] = ids.int()
    rgba[..., 3] = 255
    return dict(rgba=rgba.reshape(-1, 48, 64, 4), seg=seg.reshape(-1, 48, 64))


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return _randomized(case, seed) if case["randomize"] else _flight(case, seed)
    if kind == "rollout":
        return _flight(case, seed)
    if kind == "render":
        return _camera(case, seed)
    if kind == "network":
        return _network(_init(seed), _mlp_rows(case["rows"], _gen(seed)))
    return dict(surrogate=_surrogate, train=_train, transition=_transition, dataset=_dataset)[kind](case, seed)
