"""What is timed: passes of the Contact Dynamics library through its Python entry points.

A case is a dict with a ``kind`` and sizes.  ``prepare`` builds the packing, the
system and a checkpoint of its initial state; ``run`` restores the checkpoint
and does one pass (so that passes are alike); ``exact`` solves the same pass
with plain torch in 64 bits, in the colour order that the method prescribes,
for the plain time steps and the allocation-free detection.

Kinds:

* ``rollout``       short rollouts of a small box from a checkpoint, the step replayed from a CUDA graph
                    (parameter studies on small systems: latency and launches count);
* ``detect_noalloc`` contact detection alone, by the entry point that needs no workspace (the smallest call);
* ``static_solve``  the force network of a resting pile under a fixed lid, from zero forces to the 1e-6 residual
                    (thousands of sweeps over few contacts: the latency of a sweep counts);
* ``lid_column``    a column under a force-controlled lid, one step and the observables of it;
* ``pile_step``     warm-started steps of a loaded pile up to the sweep cap, FP64 or FP32 (the headline);
* ``domains_step``  the domain-wise update of the parallel algorithm on a pile;
* ``batch_step``    a batch of independent piles of uneven size stepped together, each to its own residual;
* ``gas_step``      steps of a 3D sphere gas, FP64 or FP32 (detection and colouring count);
* ``rollout_grad``  a differentiated rollout of settling discs, forward and backward;
* ``pyramid_grad``  the same for sliding pyramids, dominated by friction and by sweeps.
"""
import math

import numpy as np
import torch

from paper_1104_3516_gb300 import autodiff, cd
from paper_1104_3516_gb300 import workloads as W

DEV = "cuda"


def listed():
    return [
        # the 1,000-disc dilute box, 20 graph-replayed steps: the smallest system that is stepped
        {"name": "dilute_1k", "kind": "rollout", "n": 1000, "steps": 20},
        # a plug-in's detection call on a small deposit: the smallest call there is
        {"name": "detect_noalloc_5k", "kind": "detect_noalloc", "dim": 2, "n": 4999},
        # the static solve that the mixed-update scan starts from: 2,000 discs, about 10,000 sweeps
        {"name": "static_2k", "kind": "static_solve", "n": 2000},
        # the medium system of the paper's Fig. 10 with its stress and orientation profiles
        {"name": "lid_column_8k", "kind": "lid_column", "n": 8000},
        # a pile of ordinary size and odd count, FP64
        {"name": "pile_5k_f64", "kind": "pile_step", "n": 4999, "precision": "f64", "steps": 2},
        # the headline pile in both precisions: 100,000 discs, 1,000 sweeps a step
        {"name": "pile_100k_f64", "kind": "pile_step", "n": 100000, "precision": "f64", "steps": 2},
        {"name": "pile_100k_f32", "kind": "pile_step", "n": 100000, "precision": "f32", "steps": 2},
        # the paper's parallel algorithm on one GPU: 16 domains, the velocity changes summed after every sweep
        {"name": "domains_20k", "kind": "domains_step", "n": 20000, "cuts": 4},
        # many packings of 200 to 20,000 discs with their own friction, from a captured graph
        {"name": "batch_128", "kind": "batch_step", "packings": 128},
        # the largest system: a million spheres
        {"name": "gas_1m_f64", "kind": "gas_step", "n": 1000000, "precision": "f64", "steps": 4},
        # gradients of a rollout with few contacts a step, and of one that sweeps 150 times a step
        {"name": "settling_10k_grad", "kind": "rollout_grad", "n": 10000, "steps": 10},
        {"name": "pyramids_10k_grad", "kind": "pyramid_grad", "pyramids": 3334, "steps": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rollout", "detect_noalloc", "static_solve", "lid_column", "pile_step", "pile_step",
                       "domains_step", "batch_step", "gas_step", "gas_step", "rollout_grad", "pyramid_grad"])
    if kind == "rollout":
        return {"kind": kind, "n": _log_int(rng, 100, 8000), "steps": rng.randint(8, 20)}
    if kind == "detect_noalloc":
        return {"kind": kind, "dim": rng.choice([2, 3]), "n": _log_int(rng, 100, 16000)}
    if kind == "static_solve":
        return {"kind": kind, "n": _log_int(rng, 300, 2000)}
    if kind == "lid_column":
        return {"kind": kind, "n": _log_int(rng, 500, 8000)}
    if kind == "pile_step":
        return {"kind": kind, "n": _log_int(rng, 1000, 100000), "precision": rng.choice(["f64", "f32"]), "steps": 2}
    if kind == "domains_step":
        return {"kind": kind, "n": _log_int(rng, 2000, 20000), "cuts": rng.randint(2, 6)}
    if kind == "batch_step":
        return {"kind": kind, "packings": _log_int(rng, 8, 96)}
    if kind == "gas_step":
        return {"kind": kind, "n": _log_int(rng, 10000, 600000), "precision": rng.choice(["f64", "f32"]),
                "steps": rng.randint(2, 4)}
    if kind == "rollout_grad":
        return {"kind": kind, "n": _log_int(rng, 500, 10000), "steps": rng.randint(4, 10)}
    return {"kind": kind, "pyramids": _log_int(rng, 200, 3334), "steps": rng.randint(2, 4)}


def sphere_gas(seed, n, phi=0.3, vsig=0.1, mu=0.5):
    """The 3D gas of the benchmark (radii U[0.8, 1.2], random sequential addition at packing fraction 0.3, velocities
    N(0, 0.1), gravity, a floor and four side walls): a periodic block of at most 16,000 spheres is placed and
    repeated, so that a million of them take seconds."""
    tiles = max(1, int(math.ceil((n / 16000.0) ** (1.0 / 3.0))))
    nb = -(-n // tiles ** 3)
    r = W.uniform(seed, nb, 0.8, 1.2)
    side = max((float(np.sum(4.0 / 3.0 * math.pi * r ** 3)) / phi) ** (1.0 / 3.0), 12.0)
    x = W.rsa(3, nb, r, (0.0, 0.0, 0.0), (side, side, side), (1, 1, 1), seed)
    k = np.arange(tiles) * side
    shift = np.stack(np.meshgrid(k, k, k, indexing="ij"), axis=-1).reshape(-1, 3)
    x = (shift[:, None, :] + x[None, :, :]).reshape(-1, 3)[:n]
    r = np.tile(r, tiles ** 3)[:n]
    order = W.spatial_order(x, 2.4)
    x, r = np.ascontiguousarray(x[order]), np.ascontiguousarray(r[order])
    v = W.normal(seed, 3 * n, vsig).reshape(n, 3)
    inv_m, inv_I = W.masses(3, r)
    lo, hi = -1.2, tiles * side + 1.2
    return W.Workload(name="sphere_gas_3d", dim=3, x=x, v=v, w=np.zeros((n, 3)), r=r, inv_m=inv_m, inv_I=inv_I, mu=mu,
                      gravity=(0.0, 0.0, -1.0), box_lo=(lo, lo, lo), box_hi=(hi, hi, hi + 2.4), wall_mask=0b011111,
                      wall_pos=np.array([lo, hi, lo, hi, lo, hi + 2.4]), seed=seed)


def packing(case, seed):
    """The packing of a case (the first of a batch) and the keywords of its system."""
    kind = case["kind"]
    kw = {"criterion": cd.CD_CONV_GLOBAL_REL}
    if kind == "rollout":
        n = case["n"]
        wl = W.dilute_discs(seed=seed, n=n, width=max(12.0, 40.0 * math.sqrt(n / 1000.0)))
        wl.v = W.normal(seed, 2 * n, 0.05).reshape(n, 2)
        kw["use_graph"] = 1
    elif kind == "detect_noalloc":
        n = case["n"]
        wl = W.dense_biaxial_discs(seed=seed, n=n) if case["dim"] == 2 else sphere_gas(seed, n)
    elif kind == "static_solve":
        wl = W.dense_biaxial_discs(seed=seed, n=case["n"], wall_speed=0.0)
        wl.max_sweeps = 20000
        kw.update(warm_start=0, max_contacts=4 * wl.n)
    elif kind == "lid_column":
        wl = W.pressure_column(seed=seed, n=case["n"])
    elif kind == "pile_step":
        wl = W.dense_biaxial_discs(seed=seed, n=case["n"])
        kw.update(max_contacts=4 * wl.n, precision=cd.CD_FP64 if case["precision"] == "f64" else cd.CD_FP32)
    elif kind == "domains_step":
        wl = W.dense_biaxial_discs(seed=seed, n=case["n"])
        kw.update(max_contacts=4 * wl.n, domains=(case["cuts"], case["cuts"], 1))
    elif kind == "gas_step":
        wl = sphere_gas(seed, case["n"])
        kw.update(max_contacts=4 * wl.n, precision=cd.CD_FP64 if case["precision"] == "f64" else cd.CD_FP32)
    elif kind == "rollout_grad":
        wl = W.settling_discs(seed=seed, n=case["n"])
        kw.update(use_graph=1, tape_steps=case["steps"])
    elif kind == "pyramid_grad":
        wl = W.sliding_pyramids(seed=seed, n_pyramids=case["pyramids"])
        wl.max_sweeps = 150
        kw.update(use_graph=1, tape_steps=case["steps"], criterion=cd.CD_CONV_NONE)
    else:
        raise ValueError(kind)
    return wl, kw


def _contact_arrays(m):
    """Room for m contacts: pairs, normal, gap, impulse (2D), colour."""
    z = lambda shape, dtype=torch.float64: torch.zeros(shape, dtype=dtype, device=DEV)  # noqa: E731
    return [z((m, 2), torch.int32), z((m, 3)), z(m), z((m, 2)), z(m, torch.int32)]


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "stream": torch.cuda.Stream()}
    with torch.cuda.stream(state["stream"]):
        if kind == "batch_step":
            # the batched benchmark: 200 to 20,000 discs (log-uniform) and a friction of its own per packing, a captured step
            m = case["packings"]
            mu = W.uniform(seed, m, 0.1, 0.6, stream=4)
            packs = [W.settled_pile(seed=seed * 1009 + b, n=int(n), mu=float(mu[b]))
                     for b, n in enumerate(W.batch_sizes(n_packings=m))]
            state["system"] = cd.CDSystem(packs[0], batch=packs, criterion=cd.CD_CONV_GLOBAL_REL, use_graph=1,
                                          max_contacts=4 * sum(p.n for p in packs))
            state["start"] = state["system"].save_checkpoint()
        elif kind == "detect_noalloc":
            wl, _ = packing(case, seed)
            f64 = {"dtype": torch.float64, "device": DEV}
            state.update(n=wl.n, params=cd.make_params(wl), most=min(4 * wl.n, 65536),
                         pos=torch.as_tensor(np.ascontiguousarray(wl.x).reshape(-1), **f64),
                         of=[torch.as_tensor(a, **f64) for a in (wl.r, wl.inv_m, wl.inv_I)])
            state["out"] = _contact_arrays(state["most"])[:3]
        else:
            wl, kw = packing(case, seed)
            s = state["system"] = cd.CDSystem(wl, **kw)
            if kind in ("rollout_grad", "pyramid_grad"):
                state["initial"] = [s.pos.clone(), s.vel.clone(), s.omega.clone(),
                                    torch.tensor(float(wl.mu), dtype=torch.float64)]
                state["width"] = float(wl.box_hi[0] - wl.box_lo[0])
            else:
                state["start"] = s.save_checkpoint()
                if kind in ("static_solve", "domains_step"):
                    state["out"] = _contact_arrays(4 * wl.n)
    state["stream"].synchronize()
    return state


def _particles(s):
    out = {"x": s.pos, "v": s.vel, "w": s.omega}
    if s.theta is not None:
        out["theta"] = s.theta
    return out


def _counts(st):
    last = st["last"]
    return {"steps": st["steps_done"], "sweeps": st["total_sweeps"], "updates": st["total_contact_updates"],
            "contacts": last["n_contacts"], "colours": last["n_colours"], "r_avg": last["r_avg"],
            "wall_force": np.array(last["wall_force"])}


def run(state):
    case = state["case"]
    kind = case["kind"]
    with torch.cuda.stream(state["stream"]):
        if kind == "detect_noalloc":
            pairs, normal, gap = state["out"]
            nc = cd.cd_detect_contacts_noalloc(state["params"], state["n"], state["pos"], *state["of"], state["most"],
                                               pairs, normal, gap, state["stream"].cuda_stream)
            return {"contacts": nc, "pairs": pairs, "normal": normal, "gap": gap}   # rows past the contacts stay 0
        s = state["system"]
        if kind in ("rollout_grad", "pyramid_grad"):
            # the floor pressure of the last step and the mean height, as a calibration would weigh them
            x0, v0, w0, mu = (t.detach().requires_grad_(True) for t in state["initial"])
            x, v, w, force = autodiff.rollout(s, x0, v0, w0, mu, case["steps"], checkpoint_every=case["steps"],
                                              alpha=1e-10)
            loss = x.reshape(-1, 2)[:, 1].mean() + (0.5 * v * v).sum() + (force[2] / state["width"]).to(x.device)
            loss.backward()
            return {"x": x, "v": v, "w": w, "force": force, "dx": x0.grad, "dv": v0.grad, "dw": w0.grad,
                    "dmu": mu.grad, "loss": loss}
        s.load_checkpoint(state["start"])
        st = s.step(case.get("steps", 1))
        out = {**_particles(s), **_counts(st)}
        if kind == "batch_step":
            per = s.packing_stats()
            out["packing_sweeps"] = np.array([p["sweeps"] for p in per])
            out["packing_r_avg"] = np.array([p["r_avg"] for p in per])
            out["packing_force"] = np.array([p["wall_force"] for p in per])
        elif kind == "lid_column":
            out["orientation"] = s.force_orientation(18)
            out["stress"] = s.stress_profile(1, 0.0, 4.0, 64)
            out["walls"] = s.walls()
        elif kind in ("static_solve", "domains_step"):
            pairs, normal, gap, impulse, colour = state["out"]   # of the capacity: rows past the contacts stay 0
            cd.cd_get_contacts(s.handle, pairs, normal, gap, impulse, colour)
            out.update(pairs=pairs, normal=normal, gap=gap, impulse=impulse, colour=colour)
        return out


def work(case):
    """Bytes: the particle state read and written, and each contact record written, once per step.  Flops: 42 (2D) or 101
    (3D) per contact update, with the contacts per particle and the sweeps that the packings of these recipes have."""
    kind = case["kind"]
    dim, steps = (3 if kind == "gas_step" else 2), case.get("steps", 1)
    n = {"batch_step": case.get("packings", 0) * 4300, "pyramid_grad": 3 * case.get("pyramids", 0)}.get(kind) or case["n"]
    per, sweeps = {"rollout": (0.7, 2), "detect_noalloc": (1.5, 0), "static_solve": (2.2, 8000 * n / 2000.0),
                   "lid_column": (2.2, 1000), "pile_step": (2.23, 1000), "domains_step": (2.2, 1000),
                   "batch_step": (2.2, 500), "gas_step": (0.88, 2.6), "rollout_grad": (0.8, 4),
                   "pyramid_grad": (4.0 / 3.0, 400)}[kind]
    words = (7 if dim == 2 else 13) + (3 if dim == 2 else 9)
    contact = 8 + 8 * (3 + 1 + 2 + (2 if dim == 2 else 4))
    nbytes = steps * n * (8 * words + per * contact)
    return {"bytes": nbytes, "flops": steps * n * per * sweeps * (42 if dim == 2 else 101)}


# ---------------------------------------------------------------------------------------------------------------------
# The same passes in 64 bits with torch alone
# ---------------------------------------------------------------------------------------------------------------------

def _pairs_near(x, r, lo, hi, periodic, delta):
    """All pairs (a, b), a < b, with |x_b - x_a| < r_a + r_b + delta (minimum image), in ascending order."""
    n, D = x.shape
    L = hi - lo
    cells = torch.clamp(torch.floor(L / (2.0 * r.max() + delta) / (1.0 + 1e-9)), min=1.0).to(torch.int64)
    at = torch.minimum(torch.clamp(torch.floor((x - lo) / L * cells).to(torch.int64), min=0), cells - 1)
    stride = torch.ones(D, dtype=torch.int64, device=x.device)
    for k in range(1, D):
        stride[k] = stride[k - 1] * cells[k - 1]
    ids, order = torch.sort((at * stride).sum(1))
    found = []
    for off in np.ndindex(*([3] * D)):
        to = at + torch.tensor(off, device=x.device) - 1
        ok = torch.ones(n, dtype=torch.bool, device=x.device)
        for k in range(D):
            if periodic[k]:
                to[:, k] %= cells[k]
            else:
                ok &= (to[:, k] >= 0) & (to[:, k] < cells[k])
        c = (to * stride).sum(1)
        first = torch.searchsorted(ids, c)
        count = torch.where(ok, torch.searchsorted(ids, c, right=True) - first, 0)
        a = torch.repeat_interleave(torch.arange(n, device=x.device), count)
        start = torch.cumsum(count, 0) - count
        b = order[first[a] + torch.arange(a.numel(), device=x.device) - start[a]]
        keep = b > a
        a, b = a[keep], b[keep]
        d = x[b] - x[a]
        for k in range(D):
            if periodic[k]:
                d[:, k] -= L[k] * (d[:, k] > 0.5 * L[k]) - L[k] * (d[:, k] < -0.5 * L[k])
        s = r[a] + r[b] + delta
        near = (d * d).sum(1) < s * s
        found.append(torch.stack([a[near], b[near]], 1))
    return torch.cat(found)


class _Exact:
    """Plain time steps of one packing in 64 bits: the method of Sec. 2.1 in colour order."""

    def __init__(self, wl):
        dev = self.dev = DEV if torch.cuda.is_available() else "cpu"
        f = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.wl, self.D = wl, wl.dim
        self.x, self.v, self.r = f(wl.x), f(wl.v), f(wl.r)
        self.w = f(wl.w).reshape(wl.n, -1)
        self.im, self.iI = f(wl.inv_m), f(wl.inv_I)
        self.lo, self.hi = f(wl.box_lo[:wl.dim]), f(wl.box_hi[:wl.dim])
        self.wall, self.wall_vel = f(wl.wall_pos).clone(), f(np.asarray(wl.wall_vel).reshape(6, 3))
        self.theta = torch.zeros(wl.n, dtype=torch.float64, device=dev)
        self.keys = self.P = None
        self.sweeps = self.updates = 0

    def contacts(self):
        wl, n, D = self.wl, self.wl.n, self.D
        ab = [_pairs_near(self.x, self.r, self.lo, self.hi, wl.periodic, wl.delta)]
        for k in range(2 * D):
            if (wl.wall_mask >> k) & 1:
                s = 1.0 if k & 1 else -1.0
                a = torch.nonzero(s * (self.wall[k] - self.x[:, k >> 1]) - self.r < wl.delta).reshape(-1)
                ab.append(torch.stack([a, torch.full_like(a, n + k)], 1))
        ab = torch.cat(ab)
        key, order = torch.sort(ab[:, 0] * (n + 6) + ab[:, 1])
        ab = ab[order]
        a, b = ab[:, 0], ab[:, 1]
        pair = (b < n)[:, None]
        j = torch.where(b < n, b, 0)
        d = self.x[j] - self.x[a]
        for k in range(D):
            if wl.periodic[k]:
                L = self.hi[k] - self.lo[k]
                d[:, k] -= L * (d[:, k] > 0.5 * L) - L * (d[:, k] < -0.5 * L)
        dist = torch.sqrt((d * d).sum(1))
        k = torch.where(b < n, 0, b - n)
        side = torch.where(k % 2 == 1, 1.0, -1.0).to(torch.float64)
        axis = torch.nn.functional.one_hot(k // 2, 3)[:, :D].to(torch.float64)
        nrm = torch.where(pair, d / torch.clamp(dist, min=1e-300)[:, None], axis * side[:, None])
        gap_w = side * (self.wall[k] - (self.x[a] * axis).sum(1)) - self.r[a]
        gap = torch.where(b < n, dist - (self.r[a] + self.r[j]), gap_w)
        return key, ab, nrm, gap

    def colours(self, ab):
        """Greedy in descending priority (contacts of both bodies, then the hash of the key), in rounds of local maxima,
        then the alternating-path repair of the highest colour."""
        n, nc = self.wl.n, ab.shape[0]
        p = ab.cpu().numpy().astype(np.uint64)
        with np.errstate(over="ignore"):
            z = (np.uint64(self.wl.seed & (2 ** 64 - 1)) ^ (p[:, 0] << np.uint64(32) | p[:, 1])) + np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z ^= z >> np.uint64(31)
        deg = np.bincount(p.reshape(-1).astype(np.int64), minlength=n + 6)
        deg[n:] = 0
        q = p.astype(np.int64)
        prio = np.minimum(deg[q[:, 0]] + deg[q[:, 1]], 255).astype(np.uint64) << np.uint64(56) | z >> np.uint64(8)
        rank = np.empty(nc, np.int64)
        rank[np.lexsort((np.arange(nc), ~prio))] = np.arange(nc, 0, -1)
        rank = torch.as_tensor(rank, device=self.dev)
        a, b = ab[:, 0], ab[:, 1]
        body = b < n
        col = torch.full((nc,), -1, dtype=torch.int64, device=self.dev)
        used = torch.zeros(n + 6, dtype=torch.int64, device=self.dev)
        left = torch.arange(nc, device=self.dev)
        while left.numel():
            top = torch.zeros(n + 6, dtype=torch.int64, device=self.dev)
            top.scatter_reduce_(0, a[left], rank[left], "amax")
            top.scatter_reduce_(0, b[left], rank[left], "amax")
            ready = (top[a[left]] == rank[left]) & (~body[left] | (top[b[left]] == rank[left]))
            c = left[ready]
            m = used[a[c]] | torch.where(body[c], used[b[c]], 0)
            k = torch.zeros_like(c)
            while bool(((m >> k) & 1).any()):
                k += (m >> k) & 1
            col[c] = k
            used[a[c]] |= 1 << k
            at = c[body[c]]
            used[b[at]] |= 1 << k[body[c]]
            left = left[~ready]
        col = col.cpu().numpy()
        T, dmax = int(col.max(initial=-1)), int(deg.max(initial=0))
        tops = np.nonzero(col == T)[0]
        if T <= 0 or T + 1 <= dmax or len(tops) > max(1, min(1024, nc // 256)):
            return torch.as_tensor(col, device=self.dev)
        ends = np.concatenate([q[:, 0], q[:, 1]])
        order = np.argsort(ends, kind="stable")
        start, who = np.searchsorted(ends[order], np.arange(n + 7)), order % max(nc, 1)
        at = lambda x: who[start[x]:start[x + 1]]  # noqa: E731
        spare = lambda x, c: [k for k in range(T) if x >= n or k not in {int(col[e]) for e in at(x) if e != c}]  # noqa: E731
        for c in tops:
            u, v = int(q[c, 0]), int(q[c, 1])
            fu, fv = spare(u, c), spare(v, c)
            both = [k for k in fu if k in fv]
            if both or v >= n:
                col[c] = both[0] if both else T
                continue
            for i, k in [(i, k) for i in fu for k in fv]:
                path, x, cur = [], v, i
                while True:
                    e = next((int(e) for e in at(x) if col[e] == cur), -1)
                    if e < 0:
                        break
                    y = int(q[e, 0] + q[e, 1]) - x
                    path.append(e)
                    if y == u or y >= n:
                        break
                    x, cur = y, (k if cur == i else i)
                if path and int(q[path[-1], 0] + q[path[-1], 1]) - x == u:
                    continue
                for e in path:
                    col[e] = k if col[e] == i else i
                col[c] = i
                break
        return torch.as_tensor(col, device=self.dev)

    def step(self):
        wl, n, D = self.wl, self.wl.n, self.D
        key, ab, nrm, gap = self.contacts()
        nc = ab.shape[0]
        P = torch.zeros((nc, D), dtype=torch.float64, device=self.dev)   # normal, then tangential (a vector in 3D)
        if D == 3:
            P = torch.zeros((nc, 4), dtype=torch.float64, device=self.dev)
        if self.keys is not None and self.keys.numel() and nc:
            i = torch.clamp(torch.searchsorted(self.keys, key), max=self.keys.numel() - 1)
            P = torch.where((self.keys[i] == key)[:, None], self.P[i], 0.0)
            if D == 3:
                P[:, 1:] -= (P[:, 1:] * nrm).sum(1, keepdim=True) * nrm
        col = self.colours(ab) if nc else ab.new_zeros(0)
        z6 = torch.zeros(6, dtype=torch.float64, device=self.dev)
        im, iI, r = torch.cat([self.im, z6]), torch.cat([self.iI, z6]), torch.cat([self.r, z6])
        g = torch.tensor(wl.gravity[:D], dtype=torch.float64, device=self.dev)
        v = torch.cat([self.v + g * wl.dt * (self.im > 0)[:, None], self.wall_vel[:, :D]])
        w = torch.cat([self.w, torch.zeros((6, self.w.shape[1]), dtype=torch.float64, device=self.dev)])
        groups = []
        for k in range(int(col.max()) + 1 if nc else 0):
            c = torch.nonzero(col == k).reshape(-1)
            a, b = ab[c, 0], ab[c, 1]
            wn = im[a] + im[b]
            wt = wn + r[a] ** 2 * iI[a] + r[b] ** 2 * iI[b]
            groups.append((c, torch.cat([a, b]), c.numel(), nrm[c], gap[c] / wl.dt, 1.0 / wn, 1.0 / wt, r[a], r[b],
                           torch.cat([-im[a], im[b]])[:, None], torch.cat([r[a] * iI[a], r[b] * iI[b]])))

        def kick(G, dn, dt):
            c, both, m, N, _, _, _, _, _, s, rot = G
            if D == 2:
                d = dn[:, None] * N + dt[:, None] * torch.stack([-N[:, 1], N[:, 0]], 1)
                turn = torch.cat([dt, dt])[:, None]
            else:
                d = dn[:, None] * N + dt
                turn = torch.cat([torch.linalg.cross(N, d)] * 2)
            v[both] = v[both] + s * torch.cat([d, d])
            w[both] = w[both] - rot[:, None] * turn

        split = (lambda q: (q[:, 0], q[:, 1])) if D == 2 else (lambda q: (q[:, 0], q[:, 1:]))
        for G in groups:
            kick(G, *split(P[G[0]]))
        mean = lambda: float(torch.sqrt((P * P).sum(1)).mean()) if nc else 0.0  # noqa: E731
        R, done, sweeps = mean(), nc == 0, 0
        while not done and sweeps < wl.max_sweeps:
            for G in groups:
                c, both, m, N, bias, mn, mt, ra, rb, _, _ = G
                V, Q, old = v[both], w[both], P[c]
                du = V[m:] - V[:m]
                if D == 2:
                    un = (du * N).sum(1)
                    ut = du[:, 1] * N[:, 0] - du[:, 0] * N[:, 1] - (ra * Q[:m, 0] + rb * Q[m:, 0])
                    pn = torch.clamp(old[:, 0] - mn * (bias + un), min=0.0)
                    lim = wl.mu * pn
                    pt = torch.minimum(torch.maximum(old[:, 1] - mt * ut, -lim), lim)
                    new = torch.stack([pn, pt], 1)
                else:
                    u = du - torch.linalg.cross(ra[:, None] * Q[:m] + rb[:, None] * Q[m:], N)
                    un = (u * N).sum(1)
                    pn = torch.clamp(old[:, 0] - mn * (bias + un), min=0.0)
                    pt = old[:, 1:] - mt[:, None] * (u - un[:, None] * N)
                    size, lim = torch.sqrt((pt * pt).sum(1)), wl.mu * pn
                    pt = torch.where((size > lim)[:, None], pt * (lim / torch.clamp(size, min=1e-300))[:, None], pt)
                    new = torch.cat([pn[:, None], pt], 1)
                kick(G, *split(new - old))
                P[c] = new
            sweeps += 1
            last, R = R, mean()
            done = abs(R - last) < wl.alpha * (R + last) or R + last == 0.0
        self.v, self.w = v[:n], w[:n]
        self.x = self.x + self.v * wl.dt
        for k in range(D):
            if wl.periodic[k]:
                L = self.hi[k] - self.lo[k]
                self.x[:, k] += L * (self.x[:, k] < self.lo[k]) - L * (self.x[:, k] >= self.hi[k])
        if D == 2:
            self.theta = self.theta + self.w[:, 0] * wl.dt
        wall_force = np.zeros(6)
        for k in range(2 * D):
            wall_force[k] = float(P[ab[:, 1] == n + k, 0].sum()) / wl.dt
            if (wl.wall_mask >> k) & 1:
                self.wall[k] += self.wall_vel[k, k >> 1] * wl.dt
        self.keys, self.P = (None, None)
        self.sweeps += sweeps
        self.updates += sweeps * nc
        return key, P, ab, col, {"contacts": nc, "colours": len(groups), "r_avg": R, "wall_force": wall_force}


def exact(case, seed):
    kind = case["kind"]
    if kind == "detect_noalloc":
        wl, _ = packing(case, seed)
        _, ab, nrm, gap = _Exact(wl).contacts()
        m, most = ab.shape[0], min(4 * wl.n, 65536)
        pairs, normal, gaps = (torch.zeros(shape, dtype=torch.float64) for shape in ((most, 2), (most, 3), most))
        pairs[:m], normal[:m, :wl.dim], gaps[:m] = ab.cpu(), nrm.cpu(), gap.cpu()
        return {"contacts": m, "pairs": pairs.to(torch.int32), "normal": normal, "gap": gaps}
    # the other kinds have no plain restatement here (a lid that moves, domains, gradients, a batch's many solves) or take
    # too long in it (the ten thousand sweeps of a static solve)
    if kind not in ("rollout", "pile_step", "gas_step"):
        return None
    wl, _ = packing(case, seed)
    e = _Exact(wl)
    for k in range(case["steps"]):
        e.keys, e.P, _, _, last = e.step()
    out = {"x": e.x.reshape(-1), "v": e.v.reshape(-1), "w": e.w.reshape(-1)}
    if e.D == 2:
        out["theta"] = e.theta
    return {**out, "steps": case["steps"], "sweeps": e.sweeps, "updates": e.updates, **last}
