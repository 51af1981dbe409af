"""What the speed of this framework is measured on: the calls a user makes, over the range of sizes in use.

Kinds of work:
  check     collision verdicts of given configurations (start / goal selection, validation)
  esdf      a new occupancy grid becomes a distance field, which is read back or checked against
  plan      a batch of planning problems: serial, lockstep and asynchronous workers
  grads     loss and gradients of the learned sampling proposal
  train     Adam steps of the learned sampling proposal
  mixtures  inference of the learned sampling proposal for a batch of problems
  gemm      the dense layer by itself
"""
import math

import numpy as np
import torch

from paper_2503_06757_gb300 import learned as L
from paper_2503_06757_gb300 import prrtc as P
from paper_2503_06757_gb300 import workload as W

MODES = {"async": P.MODE_ASYNC, "serial": P.MODE_SERIAL, "lockstep": P.MODE_LOCKSTEP}
COMPONENTS = 8
PATH_ROWS = 128  # waypoints of the longest path a plan may return
ORIGIN = (-0.8, -0.8, 0.0)


def listed():
    return [
        # One request of a validation service: a few configurations, host in, host out.
        dict(name="check_64_host", kind="check", robot="arm7", scene="shelf", obstacles=50, n=64, host=True,
             spheres=False),
        # Rejection sampling of starts and goals on the device, a million at a time.
        dict(name="check_1m", kind="check", robot="arm7", scene="shelf", obstacles=50, n=1 << 20, host=False,
             spheres=False),
        # The two-armed robot in the most cluttered scene, with the sphere centres that the choice of goals reads;
        # a count that fills no whole block.
        dict(name="check_dual_spheres", kind="check", robot="dual14", scene="mixed", obstacles=600, n=100003,
             host=False, spheres=True),
        # The sensor loop at 2 cm voxels over the workspace: new occupancy in, distance field out.
        dict(name="esdf_80_field", kind="esdf", nx=80, ny=80, nz=80, check=0),
        # The same loop at a fine grid, where the field stays on the device and a set of states is checked against it.
        dict(name="esdf_256_check", kind="esdf", nx=256, ny=256, nz=256, check=65536),
        # Reproducible planning in the order of the serial algorithm: one worker a problem.
        dict(name="plan_serial_200", kind="plan", mode="serial", robot="arm7", scene="shelf", obstacles=50,
             problems=200, workers=1, iters=50000),
        # Reproducible planning with concurrent workers.
        dict(name="plan_lockstep_200", kind="plan", mode="lockstep", robot="arm7", scene="shelf", obstacles=50,
             problems=200, workers=8, iters=50000),
        # The fast schedule on the same problems.  Its workers race, so two runs find different paths between the same
        # ends: what can be compared is which problems were solved, and that each path runs from its start to its goal.
        dict(name="plan_async_200", kind="plan", mode="async", robot="arm7", scene="shelf", obstacles=50,
             problems=200, workers=0, iters=50000),
        # Held-out loss and gradients of the two-armed robot's proposal at its training batch.
        dict(name="grads_512", kind="grads", robot="dual14", batch=512),
        # Training: a run of optimiser steps on a set of path samples.
        dict(name="train_512", kind="train", robot="arm7", batch=512, steps=32, samples=16384, scenes=16),
        # Mixtures for a batch of problems before learned planning.
        dict(name="mixtures_300", kind="mixtures", robot="arm7", problems=300, scenes=300),
        # The dense layer where the tensor cores bound it.
        dict(name="gemm_8192", kind="gemm", m=8192, n=8192, k=8192, bias=False, relu=False, out="bf16"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["check", "check", "esdf", "esdf", "plan", "plan", "grads", "train", "mixtures", "gemm"])
    robot = rng.choice(["arm7", "arm8", "dual14"])
    if kind == "check":
        host = rng.random() < 0.3
        spheres = rng.random() < 0.4
        scene = rng.choice(["shelf", "mixed"])
        return dict(kind=kind, robot=robot, scene=scene, obstacles=50 if scene == "shelf" else _log(rng, 10, 600),
                    n=_log(rng, 1, 30000 if host else (150000 if spheres else 1 << 20)), host=host, spheres=spheres)
    if kind == "esdf":
        check = rng.choice([0, _log(rng, 1, 65536)])
        top = 128 if check == 0 else 256
        return dict(kind=kind, nx=_log(rng, 16, top), ny=_log(rng, 16, top), nz=_log(rng, 16, top), check=check)
    if kind == "plan":
        mode = rng.choice(["serial", "lockstep", "lockstep", "async"])
        if mode == "async":  # problems that every run solves
            return dict(kind=kind, mode=mode, robot="arm7", scene="shelf", obstacles=50,
                        problems=rng.randrange(32, 257), workers=0, iters=50000)
        scene = rng.choice(["shelf", "mixed"])
        return dict(kind=kind, mode=mode, robot=robot, scene=scene,
                    obstacles=50 if scene == "shelf" else _log(rng, 10, 120), problems=_log(rng, 1, 200),
                    workers=_log(rng, 2, 64) if mode == "lockstep" else 1, iters=2000)
    if kind == "grads":
        return dict(kind=kind, robot=robot, batch=_log(rng, 8, 2048))
    if kind == "train":
        return dict(kind=kind, robot=robot, batch=_log(rng, 32, 1024), steps=rng.randrange(4, 33),
                    samples=_log(rng, 1024, 16384), scenes=rng.randrange(1, 17))
    if kind == "mixtures":
        problems = _log(rng, 1, 300)
        return dict(kind=kind, robot=robot, problems=problems, scenes=_log(rng, 1, problems))
    return dict(kind=kind, m=_log(rng, 8, 8192), n=8 * _log(rng, 8, 1024), k=8 * _log(rng, 8, 1024),
                bias=rng.random() < 0.5, relu=rng.random() < 0.5, out=rng.choice(["bf16", "fp32"]))


# ----------------------------------------------------------------------------------------------- inputs

def _seed(seed):
    return 1000 + (int(seed) * 7919) % (1 << 28)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(_seed(seed))


def _scene(robot, case, seed):
    if case["scene"] == "shelf":
        return W.scene_shelf(seed, W.shelf_facing(robot))
    return W.scene_mixed(seed, case["obstacles"], bases=W.robot_bases(robot))


def _configs(robot, n, gen):
    lo = torch.tensor(robot.lower, dtype=torch.float32, device="cuda")
    hi = torch.tensor(robot.upper, dtype=torch.float32, device="cuda")
    return lo + (hi - lo) * torch.rand(n, robot.dof, generator=gen, device="cuda")


def _check_inputs(case, seed):
    robot = W.ROBOTS[case["robot"]]()
    return robot, _scene(robot, case, _seed(seed)), _configs(robot, case["n"], _gen(seed))


def _voxel(case):
    return float(np.float32(1.6 / max(case["nx"], case["ny"], case["nz"])))


def _occupancy(case, seed):
    ev = P.make_env(W.scene_shelf(_seed(seed)))
    return ev.voxelize(ORIGIN, _voxel(case), (case["nx"], case["ny"], case["nz"]))


def _pairs(robot, rb, scene, ev, n, seed, in_cells):
    if in_cells:
        s, g = L.scene_pairs(robot, scene, rb, ev, n, seed, chunk=2048, max_chunks=4)
        return list(zip(s, g))
    Q = W.candidates(robot, seed, 0, 2048).astype(np.float32)
    free = Q[P.prrtc_check_states(rb, ev, Q)]
    return [(free[2 * i], free[2 * i + 1]) for i in range(min(n, len(free) // 2))]


def _problems(case, seed):
    """Problems of several scenes, eight start / goal pairs in each."""
    robot = W.ROBOTS[case["robot"]]()
    rb = P.make_robot(robot)
    items, k = [], 0
    in_cells = case["scene"] == "shelf"
    while len(items) < case["problems"]:
        if k >= 4 * case["problems"] + 64:
            raise RuntimeError("no start / goal pairs in these scenes")
        s0 = _seed(seed) + k
        k += 1
        scene = _scene(robot, case, s0)
        ev = P.make_env(scene)
        for s, g in _pairs(robot, rb, scene, ev, min(8, case["problems"] - len(items)), s0, in_cells):
            items.append((rb, ev, s, g, s0 & 0xffff, len(items)))
    return items


def _proposal_params(robot, seed):
    """He-normal weights, and biases as they are after some training: [(W [out, in], b [out])] in FP32 on the GPU."""
    dims = (W.PROPOSAL_IN,) + W.PROPOSAL_HIDDEN + (W.proposal_head_pad(robot.dof),)
    gen = _gen(seed)
    out = []
    for i in range(4):
        scale = math.sqrt(2.0 / dims[i]) if i < 3 else 0.1 * math.sqrt(1.0 / dims[i])
        out.append((scale * torch.randn(dims[i + 1], dims[i], generator=gen, device="cuda"),
                    0.02 * torch.randn(dims[i + 1], generator=gen, device="cuda")))
    return out


def _proposal(robot, seed):
    flat = torch.cat([torch.cat([w.reshape(-1), b]) for w, b in _proposal_params(robot, seed)]).cpu().numpy()
    return P.Proposal(robot.dof, robot.lower, robot.upper, flat)


def _samples(robot, n, seed):
    """Starts, goals and targets: points on the way from start to goal, off the straight line as solution paths are."""
    gen = _gen(seed + 1)
    s, g = _configs(robot, n, gen), _configs(robot, n, gen)
    t = torch.rand(n, 1, generator=gen, device="cuda")
    x = s + t * (g - s) + 0.3 * torch.randn(n, robot.dof, generator=gen, device="cuda")
    lo = torch.tensor(robot.lower, dtype=torch.float32, device="cuda")
    hi = torch.tensor(robot.upper, dtype=torch.float32, device="cuda")
    return tuple(v.cpu().numpy() for v in (s, g, torch.minimum(torch.maximum(x, lo), hi)))


def _shelf_scenes(robot, n, seed):
    return [W.scene_shelf(_seed(seed) + i, W.shelf_facing(robot)) for i in range(n)]


def _grid_rows(robot, n, scenes, seed):
    occ = np.stack([P.prrtc_occupancy(P.make_env(sc)) for sc in _shelf_scenes(robot, scenes, seed)])
    return occ, (np.arange(n) * scenes // n).astype(np.int32)


def _gemm_inputs(case, seed):
    """Activations after a ReLU, weights of unit gain."""
    gen = _gen(seed)
    a = torch.randn(case["m"], case["k"], generator=gen, device="cuda").clamp_(min=0).to(torch.bfloat16)
    b = (torch.randn(case["n"], case["k"], generator=gen, device="cuda") * math.sqrt(2.0 / case["k"])).to(torch.bfloat16)
    bias = 0.1 * torch.randn(case["n"], generator=gen, device="cuda") if case["bias"] else None
    return a, b, bias


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind)
    if kind == "check":
        robot, scene, q = _check_inputs(case, seed)
        st.update(rb=P.make_robot(robot), ev=P.make_env(scene))
        if case["host"]:
            st["q"] = q.cpu().numpy()
        else:
            st["q"] = q
            st["valid"] = torch.zeros(case["n"], dtype=torch.uint8, device="cuda")
            st["sph"] = torch.zeros(case["n"], robot.n_spheres, 4, device="cuda") if case["spheres"] else None
    elif kind == "esdf":
        occ = _occupancy(case, seed)
        st.update(occ=occ, ev=P.Env.from_occupancy(np.zeros_like(occ), ORIGIN, _voxel(case)))
        if case["check"]:
            robot = W.arm7()
            st.update(rb=P.make_robot(robot), q=_configs(robot, case["check"], _gen(seed)),
                      valid=torch.zeros(case["check"], dtype=torch.uint8, device="cuda"))
    elif kind == "plan":
        prm = P.params(mode=MODES[case["mode"]], max_iters=case["iters"], path_capacity=PATH_ROWS)
        if case["mode"] == "lockstep":
            prm.workers = case["workers"]
        st.update(items=_problems(case, seed), prm=prm)
        st["batch"] = P.PlanBatch(st["items"])
    elif kind == "grads":
        robot = W.ROBOTS[case["robot"]]()
        occ, of = _grid_rows(robot, case["batch"], min(8, case["batch"]), seed)
        st.update(prop=_proposal(robot, seed), occ=occ[of], data=_samples(robot, case["batch"], seed))
    elif kind == "train":
        robot = W.ROBOTS[case["robot"]]()
        occ, of = _grid_rows(robot, case["samples"], case["scenes"], seed)
        st.update(prop=_proposal(robot, seed), occ=occ, of=of, data=_samples(robot, case["samples"], seed))
    elif kind == "mixtures":
        robot = W.ROBOTS[case["robot"]]()
        envs = [P.make_env(sc) for sc in _shelf_scenes(robot, case["scenes"], seed)]
        n = case["problems"]
        s, g, _ = _samples(robot, n, seed)
        st.update(prop=_proposal(robot, seed), envs=[envs[i * len(envs) // n] for i in range(n)], s=s, g=g)
    else:
        a, b, bias = _gemm_inputs(case, seed)
        kind_out = torch.bfloat16 if case["out"] == "bf16" else torch.float32
        st.update(a=a, b=b, bias=bias, c=torch.empty(case["m"], case["n"], dtype=kind_out, device="cuda"))
    return st


# ----------------------------------------------------------------------------------------------- the calls

def _stream():
    return torch.cuda.current_stream().cuda_stream


def run(state):
    case, kind = state["case"], state["kind"]
    if kind == "check":
        if case["host"]:
            r = P.prrtc_check_states(state["rb"], state["ev"], state["q"], want_spheres=case["spheres"])
            return dict(valid=r[0], spheres=r[1]) if case["spheres"] else dict(valid=r)
        P.prrtc_check_states_device(state["rb"], state["ev"], state["q"].data_ptr(), case["n"],
                                    state["valid"].data_ptr(),
                                    state["sph"].data_ptr() if case["spheres"] else 0, _stream())
        return dict(valid=state["valid"], spheres=state["sph"])
    if kind == "esdf":
        state["ev"].update_occupancy(state["occ"])
        if not case["check"]:
            return dict(field=state["ev"].esdf())
        P.prrtc_check_states_device(state["rb"], state["ev"], state["q"].data_ptr(), case["check"],
                                    state["valid"].data_ptr(), 0, _stream())
        return dict(valid=state["valid"])
    if kind == "plan":
        r = state["batch"].run(state["prm"])
        paths = np.zeros((r.n, PATH_ROWS, state["items"][0][0].dof), np.float32)
        for k in range(r.n):
            p = r.path(k)
            paths[k, :len(p)] = p
        if case["mode"] == "async":
            return dict(status=r["status"], start=paths[:, 0], goal=paths[np.arange(r.n), np.maximum(r["n"], 1) - 1])
        return dict(status=r["status"], cost=r["cost"], iterations=r["iterations"], nodes_a=r["nodes_a"],
                    nodes_b=r["nodes_b"], edges_checked=r["edges_checked"], edge_states=r["edge_states"], n=r["n"],
                    path=paths)
    if kind == "grads":
        loss, grads = state["prop"].loss_and_grads(state["occ"], *state["data"])
        return dict(loss=loss, grads=grads)
    if kind == "train":
        losses = state["prop"].train(state["occ"], state["of"], *state["data"], batch=case["batch"],
                                     steps=case["steps"], lr=1e-3, seed=5)
        return dict(losses=losses, params=state["prop"].params())
    if kind == "mixtures":
        return dict(mix=state["prop"].mixtures(state["envs"], state["s"], state["g"]))
    bf = case["out"] == "bf16"
    P.prrtc_gemm_bf16(state["a"].data_ptr(), state["b"].data_ptr(), case["m"], case["n"], case["k"],
                      state["bias"].data_ptr() if case["bias"] else 0, case["relu"],
                      0 if bf else state["c"].data_ptr(), state["c"].data_ptr() if bf else 0, _stream())
    return dict(c=state["c"])


# ----------------------------------------------------------------------------------------------- work

SPHERES = {"arm7": (28, 7, 7), "arm8": (32, 8, 8), "dual14": (56, 14, 14)}  # spheres, links, joints
STATES = {"async": 5600, "serial": 1600, "lockstep": 4500}                  # states a shelf problem has checked


def _state_flops(robot, obstacles):
    """One state: the joint chain, every sphere's centre, every link's bounding sphere against every obstacle."""
    s, links, dof = SPHERES[robot]
    return 45 * dof + 18 * s + 12 * links * obstacles


def work(case):
    kind = case["kind"]
    if kind == "check":
        s, _, dof = SPHERES[case["robot"]]
        return dict(bytes=case["n"] * (4 * dof + 1 + (16 * s if case["spheres"] else 0)),
                    flops=case["n"] * _state_flops(case["robot"], case["obstacles"]))
    if kind == "esdf":
        v = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=5 * v + 29 * case["check"], flops=3 * 4 * v + case["check"] * 28 * 40)
    if kind == "plan":
        n = case["problems"] * STATES[case["mode"]]
        return dict(bytes=case["problems"] * 4096, flops=n * _state_flops(case["robot"], case["obstacles"]))
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=2 * (m * k + n * k) + m * n * (2 if case["out"] == "bf16" else 4), flops=2 * m * n * k)
    dims = (W.PROPOSAL_IN,) + W.PROPOSAL_HIDDEN + (W.proposal_head_pad(W.ROBOTS[case["robot"]]().dof),)
    weights = sum(dims[i] * dims[i + 1] for i in range(4))
    if kind == "mixtures":
        return dict(bytes=2 * weights + case["problems"] * 4 * dims[4], flops=2 * weights * case["problems"])
    # forward, input gradients of all layers but the first, weight gradients
    flops = 2 * case["batch"] * (3 * weights - dims[0] * dims[1])
    if kind == "grads":
        return dict(bytes=6 * weights + case["batch"] * 4096, flops=flops)
    # an optimiser step reads and writes the FP32 weights and both moments and writes the BF16 weights
    return dict(bytes=case["steps"] * 30 * weights, flops=case["steps"] * flops)


# ----------------------------------------------------------------------------------------------- in 64 bits

def _fk64(robot, q):
    """World centres [n, spheres, 3] of the sphere model."""
    n = q.shape[0]
    out = torch.zeros(n, robot.n_spheres, 3, dtype=torch.float64, device=q.device)
    off = torch.tensor(np.asarray(robot.sphere_offset, np.float32), dtype=torch.float64, device=q.device)
    R = p = None
    for i in range(robot.dof):
        if robot.joint_parent[i] < 0:
            R = torch.eye(3, dtype=torch.float64, device=q.device).expand(n, 3, 3)
            base = torch.tensor(np.asarray(robot.joint_base[i], np.float32), dtype=torch.float64, device=q.device)
            p = base.expand(n, 3)
        ty, x = int(robot.joint_type[i]), q[:, i]
        if ty in W.PRISMATIC:
            axis = {W.JOINT_PRISM_X: 0, W.JOINT_PRISM_Y: 1, W.JOINT_PRISM_Z: 2}[ty]
            p = p + R[:, :, axis] * x[:, None]
        else:
            a = {W.JOINT_REV_X: 0, W.JOINT_REV_Y: 1, W.JOINT_REV_Z: 2}[ty]
            b, c = (a + 1) % 3, (a + 2) % 3
            J = torch.zeros(n, 3, 3, dtype=torch.float64, device=q.device)
            J[:, a, a] = 1
            J[:, b, b] = J[:, c, c] = torch.cos(x)
            J[:, c, b], J[:, b, c] = torch.sin(x), -torch.sin(x)
            R = R @ J
        p = p + R[:, :, 2] * float(np.float32(robot.link_length[i]))
        for s in np.nonzero(np.asarray(robot.sphere_frame) == i)[0]:
            out[:, s] = (R @ off[s]) + p
    return out


def _edt2(occ, axis, f):
    """min over t of f(t) + (i - t)^2 along one axis."""
    n = occ.shape[axis]
    i = torch.arange(n, device=f.device)
    best = torch.full_like(f, 1 << 40)
    view = [1, 1, 1]
    view[axis] = n
    for t in range(n):
        best = torch.minimum(best, f.narrow(axis, t, 1) + ((i - t) ** 2).reshape(view))
    return best


def _field64(occ, voxel):
    o = torch.tensor(occ, device="cuda") != 0
    d2 = []
    for sites in (o, ~o):
        f = torch.where(sites, 0, 1 << 40)
        for axis in (2, 1, 0):
            f = _edt2(occ, axis, f)
        d2.append(f)
    diag = voxel * math.sqrt(sum(float(d) ** 2 for d in occ.shape))
    d = torch.where(o, d2[1], d2[0])
    mag = torch.where(d >= (1 << 39), torch.full_like(d, diag, dtype=torch.float64), voxel * d.double().sqrt())
    return torch.where(o, -mag, mag)


def _grid64(scene):
    """Coarse occupancy: centres closer than 5 cm to an obstacle."""
    g = torch.arange(16, dtype=torch.float64, device="cuda")
    k, j, i = torch.meshgrid(g, g, g, indexing="ij")
    p = torch.stack([ORIGIN[a] + 0.1 * (v + 0.5) for a, v in ((0, i), (1, j), (2, k))], -1).reshape(-1, 1, 3)
    t = lambda x: torch.tensor(np.asarray(x, np.float32), dtype=torch.float64, device="cuda")
    d2 = []
    if len(scene.boxes):
        b = t(scene.boxes)
        local = torch.einsum("boj,ojk->bok", p - b[:, 0:3], b[:, 6:15].reshape(-1, 3, 3))
        d2.append(((local.abs() - b[:, 3:6]).clamp(min=0) ** 2).sum(-1))
    if len(scene.cylinders):
        c = t(scene.cylinders)
        v = p - c[:, 0:3]
        z = (v * c[:, 3:6]).sum(-1)
        rho = (v - z[..., None] * c[:, 3:6]).norm(dim=-1)
        d2.append((rho - c[:, 6]).clamp(min=0) ** 2 + (z.abs() - c[:, 7]).clamp(min=0) ** 2)
    if len(scene.spheres):
        s = t(scene.spheres)
        d2.append(((p - s[:, 0:3]).norm(dim=-1) - s[:, 3]).clamp(min=0) ** 2)
    return (torch.cat(d2, 1).amin(1) < 0.05 ** 2).double()


def _rows64(robot, occ, s, g):
    lo = torch.tensor(robot.lower, dtype=torch.float64, device="cuda")
    span = torch.tensor(robot.upper, dtype=torch.float64, device="cuda") - lo
    x = torch.zeros(len(s), W.PROPOSAL_IN, dtype=torch.float64, device="cuda")
    x[:, :4096] = occ
    for at, q in ((4096, s), (4128, g)):
        x[:, at:at + robot.dof] = 2 * (torch.tensor(q, dtype=torch.float64, device="cuda") - lo) / span - 1
    return x, lo, span


def _forward64(params, x):
    for i, (w, b) in enumerate(params):
        x = x @ w.T + b
        x = x.relu() if i < 3 else x
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "check":
        if not case["spheres"]:
            return None
        robot, _, q = _check_inputs(case, seed)
        c = _fk64(robot, q.double())
        r = torch.tensor(np.asarray(robot.sphere_radius, np.float32), dtype=torch.float64, device="cuda")
        return dict(valid=None, spheres=torch.cat([c, r.expand(c.shape[0], -1)[..., None]], -1))
    if kind == "esdf":
        return None if case["check"] else dict(field=_field64(_occupancy(case, seed), _voxel(case)))
    if kind == "gemm":
        a, b, bias = _gemm_inputs(case, seed)
        c = a.double() @ b.double().T
        c = c + bias.double() if case["bias"] else c
        return dict(c=c.relu() if case["relu"] else c)
    if kind == "mixtures":
        robot = W.ROBOTS[case["robot"]]()
        n, dof = case["problems"], robot.dof
        grids = torch.stack([_grid64(sc) for sc in _shelf_scenes(robot, case["scenes"], seed)])
        s, g, _ = _samples(robot, n, seed)
        at = torch.tensor([i * case["scenes"] // n for i in range(n)], device="cuda")
        x, _, _ = _rows64(robot, grids[at], s, g)
        y = _forward64([(w.double(), b.double()) for w, b in _proposal_params(robot, seed)], x)
        k = COMPONENTS * dof
        return dict(mix=torch.cat([y[:, :COMPONENTS + k], y[:, COMPONENTS + k:COMPONENTS + 2 * k].clamp(-5, 2)], 1))
    if kind == "grads":
        robot = W.ROBOTS[case["robot"]]()
        n, dof = case["batch"], robot.dof
        scenes = min(8, n)
        grids = torch.stack([_grid64(sc) for sc in _shelf_scenes(robot, scenes, seed)])
        s, g, target = _samples(robot, n, seed)
        at = torch.tensor([i * scenes // n for i in range(n)], device="cuda")
        x, lo, span = _rows64(robot, grids[at], s, g)
        params = [(w.double().requires_grad_(), b.double().requires_grad_()) for w, b in _proposal_params(robot, seed)]
        y = _forward64(params, x)
        k = COMPONENTS * dof
        mean = y[:, COMPONENTS:COMPONENTS + k].reshape(n, COMPONENTS, dof)
        ls = y[:, COMPONENTS + k:COMPONENTS + 2 * k].clamp(-5, 2).reshape(n, COMPONENTS, dof)
        u = 2 * (torch.tensor(target, dtype=torch.float64, device="cuda") - lo) / span - 1
        lp = (-0.5 * ((u[:, None] - mean) * torch.exp(-ls)) ** 2 - ls - 0.5 * math.log(2 * math.pi)).sum(-1)
        loss = -torch.logsumexp(torch.log_softmax(y[:, :COMPONENTS], 1) + lp, 1).mean()
        grads = torch.autograd.grad(loss, [v for pair in params for v in pair])
        return dict(loss=float(loss.detach()), grads=torch.cat([v.reshape(-1) for v in grads]))
    return None  # plans and runs of optimiser steps: what a rounding changes early, every later step carries on
