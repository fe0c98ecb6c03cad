"""The calls whose time this library is judged by, each through the public binding
(paper_2412_01733_gb300.treegb and .autograd), from one small cluster to the galaxy of
10^8 particles.

A case is a plain dict.  "kind" says which call a pass makes:

  accel     Workspace.accel: accelerations and potentials of (x, m)
  step      Workspace.leapfrog_step followed by Workspace.diagnostics, as a simulation loop makes them
  host      Workspace.leapfrog_step_host: the same step on a state in pinned host memory
  ensemble  Workspace.graph_launch: one captured step (with diagnostics) of many independent systems
  vjp       build, moments, forces(lists_only=True), forces_adjoint: one force evaluation's gradient
  grad      autograd.tree_leapfrog, K steps, and the backward pass of its loss
  direct    Workspace.direct: the direct sum of Eq. 1 for a sample of targets

The other entries are the particle model and count and the tree parameters.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_01733_gb300 import inputs, treegb
from paper_2412_01733_gb300.autograd import tree_leapfrog


def _case(name, kind, n, **kw):
    c = dict(name=name, kind=kind, model="plummer", n=n, precision="f32", theta=0.7, eps=0.01, order=2, leaf_cap=16,
             group_size=32)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the force on one star cluster of the ensemble's lowest size; odd size
        _case("accel_cluster_1031", "accel", 1031, theta=0.6),
        # a step of the plain reference configuration: FP64, monopole cells
        _case("step_f64_mono_16384", "step", 16384, precision="f64", order=0, tau=0.01),
        # a step of an ordinary single cluster; ragged size
        _case("step_cluster_30011", "step", 30011, tau=0.005),
        # the same-GPU FP64 force with quadrupoles that the FP32 forces are held against
        _case("accel_f64_131071", "accel", 131071, precision="f64"),
        # the opening-angle sweep's model and size, at its accurate end
        _case("accel_theta05_1048576", "accel", 1048576, theta=0.5, eps=0.005),
        # a state that lives on the host between steps
        _case("host_step_1000003", "host", 1000003, eps=0.005, tau=0.005),
        # an ordinary galaxy; ragged size
        _case("step_galaxy_10000019", "step", 10000019, model="galaxy", eps=0.02, tau=0.005),
        # the largest: the benchmark's galaxy
        _case("step_galaxy_100000000", "step", 100000000, model="galaxy", eps=0.02, tau=0.005),
        # the ensemble of 512 clusters (1024 to 65536 particles each), one captured step
        _case("ensemble_512", "ensemble", 512, model="ensemble", theta=0.6, tau=0.005, nmin=1024, nmax=65536),
        # the gradient of one force evaluation at the adjoint configuration's size
        _case("vjp_262144", "vjp", 262144),
        # a gradient step through four leapfrog steps (checkpoints every four)
        _case("grad_4_steps_65536", "grad", 65536, tau=0.01, steps=4),
        # the force-error reference: a direct sum on a sample of the sweep's particles
        _case("direct_8192_of_1048576", "direct", 1048576, eps=0.005, targets=8192),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["accel", "accel", "step", "step", "step", "host", "ensemble", "vjp", "grad", "direct"])
    c = _case("", kind, 0, theta=round(rng.uniform(0.4, 1.0), 2), eps=round(rng.uniform(0.005, 0.03), 4),
              leaf_cap=rng.choice([16, 16, 16, 8]), group_size=rng.choice([32, 32, 32, 16, 64]))
    del c["name"]
    if kind in ("accel", "step"):
        c["precision"] = rng.choice(["f32", "f32", "f32", "f64"])
        c["order"] = rng.choice([2, 2, 2, 0])
        c["model"] = rng.choice(["plummer", "galaxy"])
        c["n"] = _logint(rng, 1000, 3.0e7 if c["precision"] == "f32" else 2.0e5)
    elif kind == "host":
        c["model"] = rng.choice(["plummer", "galaxy"])
        c["n"] = _logint(rng, 2.0e5, 5.0e6)
    elif kind == "ensemble":
        c.update(model="ensemble", n=_logint(rng, 8, 512), nmin=1024, nmax=_logint(rng, 4096, 65536))
    elif kind == "vjp":
        c["precision"] = rng.choice(["f32", "f32", "f32", "f64"])
        c["order"] = rng.choice([2, 2, 0])
        c["n"] = _logint(rng, 4096, 300000 if c["precision"] == "f32" else 60000)
    elif kind == "grad":
        c["n"], c["steps"] = _logint(rng, 4096, 130000), rng.choice([2, 3, 4])
    else:
        c["precision"] = rng.choice(["f32", "f32", "f64"])
        c["n"] = _logint(rng, 1.0e5, 4.0e6)
        c["targets"] = _logint(rng, 500, 16384 if c["precision"] == "f32" else 2048)
    if kind in ("step", "host", "ensemble", "grad"):
        c["tau"] = round(rng.uniform(0.002, 0.01), 4)
    return c


# ---------------------------------------------------------------- preparation
def _dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _particles(case, seed):
    """(x, v, m, offsets or None) in the case's precision; the same values for a seed.  The clusters' sizes belong to
    the ensemble, not to the seed."""
    dev, dt = _device(), _dtype(case)
    if case["model"] == "ensemble":
        sizes = inputs.cluster_sizes(case["n"], nmin=case["nmin"], nmax=case["nmax"])
        sets = [inputs.plummer(int(k), seed + 1 + b, device=dev, dtype=dt) for b, k in enumerate(sizes)]
        x, v, m = torch.cat([t[0] for t in sets], 1), torch.cat([t[1] for t in sets], 1), torch.cat([t[2] for t in sets])
        off = np.concatenate(([0], np.cumsum(sizes))).astype(np.int64)
    elif case["model"] == "galaxy":
        (x, v, m), off = inputs.galaxy(case["n"], seed, device=dev, dtype=dt), None
    else:
        (x, v, m), off = inputs.plummer(case["n"], seed, device=dev, dtype=dt), None
    return x.contiguous(), v.contiguous(), m.contiguous(), off


def _cotangents(case, n, seed):
    """Cotangents of accelerations and potentials: of the order of the quantities' own scatter."""
    g = torch.Generator(device=_device())
    g.manual_seed(seed + 77)
    f = lambda *s: torch.randn(s, generator=g, device=_device(), dtype=torch.float64).to(_dtype(case))
    return f(3, n), 0.1 * f(n)


def _targets(case, seed):
    """A sample of particles without repetition (the particles are in random order already)."""
    n, nt = case["n"], case["targets"]
    return (torch.arange(nt, device=_device(), dtype=torch.int64) * (n // nt) + seed % (n // nt)).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    x, v, m, off = _particles(case, seed)
    n = x.shape[1]
    ws = treegb.Workspace(1 if kind == "direct" else n, G=1.0, eps=case["eps"], theta=case["theta"],
                          order=case["order"], leaf_cap=case["leaf_cap"], group_size=case["group_size"],
                          precision=case["precision"])
    s = dict(case=case, ws=ws, x=x, v=v, m=m)
    if kind == "accel":
        s["a"], s["phi"] = torch.empty_like(x), torch.empty_like(m)
    elif kind in ("step", "host", "ensemble"):
        if off is not None:
            ws.set_segments(off)
        s["a"], s["phi"] = ws.accel(x, m)  # the simulation starts from the forces at its first positions
        s["diag"] = torch.empty(8, dtype=torch.float64, device="cuda")
        if kind == "ensemble":
            ws.graph_capture(x, v, m, s["a"], case["tau"], phi=s["phi"], diag=s["diag"])
        elif kind == "host":
            for k in ("x", "v", "m", "a", "phi", "diag"):
                s[k] = s[k].cpu().pin_memory()
    elif kind == "vjp":
        s["a_bar"], s["phi_bar"] = _cotangents(case, n, seed)
    elif kind == "grad":
        s["w"] = _cotangents(case, n, seed)[0]
        for k in ("x", "v", "m"):
            s[k].requires_grad_(True)
    elif kind == "direct":
        s["targets"] = _targets(case, seed)
    torch.cuda.synchronize()
    return s


def run(s):
    c, ws = s["case"], s["ws"]
    kind = c["kind"]
    if kind == "accel":
        ws.accel(s["x"], s["m"], a=s["a"], phi=s["phi"])
        return s["a"], s["phi"]
    if kind == "step":
        ws.leapfrog_step(s["x"], s["v"], s["m"], s["a"], c["tau"], phi=s["phi"])
        ws.diagnostics(s["x"], s["v"], s["m"], s["phi"], out=s["diag"])
        return s["x"], s["v"], s["a"], s["phi"], s["diag"]
    if kind == "host":
        ws.leapfrog_step_host(s["x"], s["v"], s["m"], s["a"], c["tau"], phi=s["phi"], diag=s["diag"])
        torch.cuda.current_stream().synchronize()  # the host arrays may be read only then
        return s["x"], s["v"], s["a"], s["phi"], s["diag"]
    if kind == "ensemble":
        ws.graph_launch()
        return s["x"], s["v"], s["a"], s["phi"], s["diag"]
    if kind == "vjp":
        ws.build(s["x"])
        ws.moments(s["x"], s["m"])
        ws.forces(lists_only=True)
        return ws.forces_adjoint(s["a_bar"], s["phi_bar"])
    if kind == "grad":
        xk, vk, w = tree_leapfrog(s["x"], s["v"], s["m"], ws, c["steps"], c["tau"], 4)
        gx, gv, gm = torch.autograd.grad((xk * xk).sum() + (vk * s["w"]).sum() + w.to(xk.dtype),
                                         (s["x"], s["v"], s["m"]))
        return xk.detach(), vk.detach(), w.detach(), gx, gv, gm
    return ws.direct(s["x"], s["m"], s["targets"])


# ---------------------------------------------------------------- the work a pass cannot do without
def work(case):
    """Bytes: each input read and each output written once.  Flops: 20 per particle pair, 60 per particle and
    quadrupole cell (20 per monopole cell).  The interactions of a particle follow the opening angle and the tree's
    depth: 95 log2(n) / theta^2, three in ten of them pairs, describes the Plummer spheres (4180 at 2^20 and
    theta = 0.7, 11500 at theta = 0.4) and the galaxy of 10^8 (4760 at 0.7) to a tenth."""
    kind, e = case["kind"], 8 if case["precision"] == "f64" else 4
    if kind == "ensemble":
        n = int(inputs.cluster_sizes(case["n"], nmin=case["nmin"], nmax=case["nmax"]).sum())
        each = n / case["n"]
    else:
        n = each = case["n"]
    if kind == "direct":
        return {"bytes": 4 * e * n + 8 * case["targets"] + 32 * case["targets"], "flops": 20 * n * case["targets"]}
    pairs = min(each, 95 * math.log2(each) / case["theta"] ** 2)
    force = n * pairs * (0.3 * 20 + 0.7 * (60 if case["order"] == 2 else 20))
    if kind == "accel":
        return {"bytes": 8 * e * n, "flops": force}
    if kind in ("step", "host", "ensemble"):
        return {"bytes": 20 * e * n, "flops": force}
    if kind == "vjp":  # both sides' derivatives: about three times a force evaluation
        return {"bytes": 12 * e * n, "flops": 3 * force}
    k = case["steps"]
    return {"bytes": 24 * e * n, "flops": (k + 1) * force + k * force + (k + 1) * 3 * force}


# ---------------------------------------------------------------- the same results in 64 bits, plain torch
_BITS = 21


def _spread3(v):
    for s, k in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F), (4, 0x10C30C30C30C30C3),
                 (2, 0x1249249249249249)):
        v = (v | (v << s)) & k
    return v


def _segments(starts, end):
    """First indices of consecutive runs -> their lengths."""
    return torch.diff(torch.cat((starts, starts.new_tensor([end]))))


class _Tree:
    """The canonical tree of positions x (3, n): key order, breadth-first cells, walk groups."""

    def __init__(self, x, case):
        dev, n = x.device, x.shape[1]
        lcap, gs, delta = case["leaf_cap"], case["group_size"], 3
        x64 = x.double()
        lo, hi = x64.amin(1), x64.amax(1)
        ext = float((hi - lo).amax())
        self.k = math.frexp(ext)[1] if ext > 0 else 0
        q = torch.floor((x64 - lo[:, None]) * 2.0 ** (_BITS - self.k)).clamp(0, 2 ** _BITS - 1).long()
        key = (_spread3(q[0]) << 2) | (_spread3(q[1]) << 1) | _spread3(q[2])
        self.key, self.perm = torch.sort(key, stable=True)
        self.q = q[:, self.perm]
        key, ar = self.key, torch.arange(n, device=dev)
        first, count = torch.zeros(1, dtype=torch.long, device=dev), torch.full((1,), n, device=dev)
        F, C, L, CH, NCH, base = [], [], [], [], [], 0
        lev_of = torch.full((n,), -1, dtype=torch.long, device=dev)
        self.levels = []
        pops = []  # per level: population of each particle's cell there (0: no such cell)
        for lev in range(_BITS + 1):
            nl = first.numel()
            if nl == 0:
                break
            internal = (count > lcap) & (lev < _BITS)
            owner = torch.searchsorted(first, ar, right=True) - 1
            inside = (owner >= 0) & (ar < first[owner.clamp(min=0)] + count[owner.clamp(min=0)])
            pops.append(torch.where(inside, count[owner.clamp(min=0)], torch.zeros_like(ar)))
            self.levels.append((base, owner, inside))
            leafp = inside & ~internal[owner.clamp(min=0)]
            lev_of[leafp] = lev
            if lev < _BITS:
                sh = 3 * (_BITS - 1 - lev)
                flag = torch.ones(n, dtype=torch.bool, device=dev)
                flag[1:] = (key[1:] >> sh) != (key[:-1] >> sh)
                runs = torch.nonzero(flag).flatten()
                rlen = _segments(runs, n)
                keep = (inside & internal[owner.clamp(min=0)])[runs]
                nf, nc, par = runs[keep], rlen[keep], owner[runs[keep]]
            else:
                nf, nc, par = first[:0], count[:0], first[:0]
            nch = torch.zeros(nl, dtype=torch.long, device=dev).index_add_(0, par, torch.ones_like(par))
            F.append(first); C.append(count); NCH.append(nch)
            L.append(torch.full((nl,), lev, device=dev))
            CH.append(base + nl + torch.cumsum(nch, 0) - nch)
            base += nl
            first, count = nf, nc
        self.first, self.count, self.level = torch.cat(F), torch.cat(C), torch.cat(L)
        self.child, self.nchild = torch.cat(CH), torch.cat(NCH)
        self.corner = (self.q[:, self.first] >> (_BITS - self.level)) << (_BITS - self.level)
        # walk groups: chunks of gs, cut where neighbours sit in cells too far apart or too populous
        d = key[1:] ^ key[:-1]
        bits = torch.floor(torch.log2(d.clamp(min=1).double())).long()
        bits = bits - ((d >> bits.clamp(0, 62)) == 0).long()  # a rounded-up logarithm
        shared = torch.where(d == 0, torch.full_like(d, _BITS), torch.div(62 - bits, 3, rounding_mode="floor"))
        at = torch.minimum(shared, lev_of[1:])
        pop = self._pick(pops, at)
        start = (ar % gs) == 0
        cut = (shared < torch.maximum(lev_of[1:], lev_of[:-1]) - delta) | (pop > 128 * gs)
        start[1:] |= cut
        self.gfirst = torch.nonzero(start).flatten()
        self.gcount = _segments(self.gfirst, n)

    @staticmethod
    def _pick(pops, at):
        out = torch.zeros_like(at)
        for lev, p in enumerate(pops):
            out = torch.where(at == lev, p[1:], out)
        return out

    def centres(self, lo):
        unit = 2.0 ** (self.k - _BITS)
        half = 0.5 * 2.0 ** (_BITS - self.level).double()
        return lo[:, None] + (self.corner.double() + half) * unit

    def moments(self, xs, ms):
        """M, R (3, c), Q (6, c: xx yy zz xy xz yz) of every cell, from its own particles; differentiable."""
        c = self.centres(xs.detach().amin(1))
        c = c.detach()
        nn = self.first.numel()
        sums = torch.zeros((10, nn), dtype=torch.float64, device=xs.device)
        for base, owner, inside in self.levels:
            idx = torch.nonzero(inside).flatten()
            cell = base + owner[idx]
            u, m = xs[:, idx] - c[:, cell], ms[idx]
            rows = torch.stack((m, *(m * u), m * u[0] * u[0], m * u[1] * u[1], m * u[2] * u[2], m * u[0] * u[1],
                                m * u[0] * u[2], m * u[1] * u[2]))
            sums = sums.index_add(1, cell, rows)
        M = sums[0]
        S = sums[1:4] / M
        T = sums[4:] - M * torch.stack((S[0] * S[0], S[1] * S[1], S[2] * S[2], S[0] * S[1], S[0] * S[2], S[1] * S[2]))
        tr = T[0] + T[1] + T[2]
        Q = torch.cat((3.0 * T[:3] - tr, 3.0 * T[3:]))
        return M, c + S, Q

    def lists(self, theta, g0, g1):
        """(group, cell) of the far cells and (group, leaf) of the near leaves of groups [g0, g1)."""
        dev = self.key.device
        gf, gc = self.gfirst[g0:g1], self.gcount[g0:g1]
        gid = torch.repeat_interleave(torch.arange(g1 - g0, device=dev), gc)
        qq = self.q[:, int(gf[0]): int(gf[-1] + gc[-1])]
        glo = torch.full((3, g1 - g0), 2 ** 22, device=dev).scatter_reduce(1, gid.expand(3, -1), qq, "amin")
        ghi = torch.zeros((3, g1 - g0), dtype=torch.long, device=dev).scatter_reduce(1, gid.expand(3, -1), qq, "amax") + 1
        g, node = torch.arange(g1 - g0, device=dev), torch.zeros(g1 - g0, dtype=torch.long, device=dev)
        pc, pp = [], []
        while g.numel():
            s = 2 ** (_BITS - self.level[node])
            lo = self.corner[:, node]
            gap = torch.maximum(lo - ghi[:, g], glo[:, g] - (lo + s)).clamp(min=0)
            far = (s * s).double() < (theta * theta) * (gap * gap).sum(0).double()
            leaf = self.nchild[node] == 0
            pc.append((g[far], node[far]))
            near = ~far & leaf
            pp.append((g[near], node[near]))
            op = ~far & ~leaf
            go, no = g[op], node[op]
            k = self.nchild[no]
            g = torch.repeat_interleave(go, k)
            node = torch.repeat_interleave(self.child[no] - (torch.cumsum(k, 0) - k), k) + torch.arange(g.numel(), device=dev)
        cat = lambda z: (torch.cat([a for a, _ in z]), torch.cat([b for _, b in z]))
        return cat(pc), cat(pp)


def _pc(y, M, Q, eps2):
    """Field of cells (M, Q) at offset y from their centres: acceleration (3, ...) and potential."""
    r2 = y[0] * y[0] + y[1] * y[1] + y[2] * y[2] + eps2
    i1 = r2 ** -0.5
    i2 = i1 * i1
    i3 = i1 * i2
    if Q is None:
        return -M * i3 * y, -M * i1
    Qy = torch.stack((Q[0] * y[0] + Q[3] * y[1] + Q[4] * y[2], Q[3] * y[0] + Q[1] * y[1] + Q[5] * y[2],
                      Q[4] * y[0] + Q[5] * y[1] + Q[2] * y[2]))
    yQy = y[0] * Qy[0] + y[1] * Qy[1] + y[2] * Qy[2]
    i5 = i3 * i2
    return (-M * i3 - 2.5 * yQy * i5 * i2) * y + i5 * Qy, -M * i1 - 0.5 * yQy * i5


def _tree_field(tree, case, visit, budget=1 << 25):
    """Calls visit(rows, targets, sources, is_cell) for blocks of (entry, target) pairs of all groups: targets
    (e, gs) sorted positions with -1 where a group is shorter, sources (e) cells or sorted positions, rows (e) the
    entry's group within [g0, g1)."""
    dev = tree.key.device
    gs, ng = case["group_size"], tree.gfirst.numel()
    per = max(1, min(ng, int(3.0e7 / (200 + 95 * math.log2(tree.key.numel() + 2) / max(case["theta"], 0.1) ** 2))))
    lane = torch.arange(gs, device=dev)
    for g0 in range(0, ng, per):
        g1 = min(ng, g0 + per)
        (pg, pcell), (lg, leaf) = tree.lists(case["theta"], g0, g1)
        k = tree.count[leaf]
        lg = torch.repeat_interleave(lg, k)
        src = torch.repeat_interleave(tree.first[leaf] - (torch.cumsum(k, 0) - k), k) + torch.arange(lg.numel(), device=dev)
        for rows, ent, is_cell in ((pg, pcell, True), (lg, src, False)):
            order = torch.argsort(rows)
            rows, ent = rows[order], ent[order]
            step = max(1, budget // gs)
            for b in range(0, rows.numel(), step):
                r = rows[b: b + step]
                t = tree.gfirst[g0 + r][:, None] + lane
                t = torch.where(lane < tree.gcount[g0 + r][:, None], t, torch.full_like(t, -1))
                visit(g0 + r, t, ent[b: b + step], is_cell)


def _pair_field(t, ent, is_cell, xs, ms, mom, case):
    eps2 = case["eps"] ** 2
    p = xs[:, t.clamp(min=0)]
    ok = t >= 0
    if is_cell:
        M, R, Q = mom
        a, f = _pc(p - R[:, ent][:, :, None], M[ent][:, None], Q[:, ent][:, :, None] if case["order"] == 2 else None, eps2)
    else:
        ok = ok & (t != ent[:, None])
        a, f = _pc(p - xs[:, ent][:, :, None], ms[ent][:, None], None, eps2)
    return torch.where(ok, a, torch.zeros_like(a)), torch.where(ok, f, torch.zeros_like(f))


def _exact_accel(x, m, case):
    """Accelerations (3, n) and potentials (n) of the tree force in 64 bits, in the caller's order."""
    n, gs = x.shape[1], case["group_size"]
    tree = _Tree(x, case)
    xs, ms = x.double()[:, tree.perm], m.double()[tree.perm]
    mom = tree.moments(xs, ms)
    out = torch.zeros((4, n + 1), dtype=torch.float64, device=x.device)

    def visit(rows, t, ent, is_cell):
        a, f = _pair_field(t, ent, is_cell, xs, ms, mom, case)
        v = torch.cat((a, f[None])).permute(1, 0, 2).reshape(rows.numel(), 4 * gs)
        grp, num = torch.unique_consecutive(rows, return_counts=True)
        tot = torch.segment_reduce(v.contiguous(), "sum", lengths=num, axis=0).reshape(-1, 4, gs)
        lane = torch.arange(gs, device=x.device)
        dst = torch.where(lane < tree.gcount[grp][:, None], tree.gfirst[grp][:, None] + lane, torch.full_like(lane, n))
        out.index_add_(1, dst.flatten(), tot.permute(1, 0, 2).reshape(4, -1))

    _tree_field(tree, case, visit)
    res = torch.empty((4, n), dtype=torch.float64, device=x.device)
    res[:, tree.perm] = out[:, :n]
    return res[:3], res[3]


def _exact_vjp(x, m, a_bar, phi_bar, case):
    """Gradients (x_bar (3, n), m_bar (n)) of sum a_bar a + phi_bar phi with the tree's structure held fixed."""
    tree = _Tree(x, case)
    xs = x.double()[:, tree.perm].requires_grad_(True)
    ms = m.double()[tree.perm].requires_grad_(True)
    ab, fb = a_bar.double()[:, tree.perm], phi_bar.double()[tree.perm]
    mom = tree.moments(xs, ms)
    cut = [t.detach().requires_grad_(True) for t in mom]
    xd, md = xs.detach().requires_grad_(True), ms.detach().requires_grad_(True)

    def visit(rows, t, ent, is_cell):
        with torch.enable_grad():
            a, f = _pair_field(t, ent, is_cell, xd, md, cut, case)
            i = t.clamp(min=0)
            ((a * ab[:, i]).sum() + (f * fb[i]).sum()).backward()

    _tree_field(tree, case, visit, budget=1 << 22)
    gx, gm = torch.autograd.grad(mom, (xs, ms), grad_outputs=[c.grad if c.grad is not None else torch.zeros_like(c)
                                                              for c in cut])
    gx, gm = gx + xd.grad, gm + md.grad
    ox, om = torch.empty_like(gx), torch.empty_like(gm)
    ox[:, tree.perm], om[tree.perm] = gx, gm
    return ox, om


def _exact_direct(x, m, targets, case):
    n = x.shape[1]
    x64, m64, eps2 = x.double(), m.double(), case["eps"] ** 2
    nt = targets.numel()
    out = torch.zeros((4, nt), dtype=torch.float64, device=x.device)
    step = max(1, (1 << 26) // nt)
    for j in range(0, n, step):
        src = torch.arange(j, min(n, j + step), device=x.device)
        a, f = _pc(x64[:, targets][:, :, None] - x64[:, None, src], m64[src][None], None, eps2)
        own = targets[:, None] == src[None]
        out[:3] += torch.where(own, torch.zeros_like(a), a).sum(2)
        out[3] += torch.where(own, torch.zeros_like(f), f).sum(1)
    return out[:3], out[3]


def _exact_diag(x, v, m, phi):
    p = (m * v).sum(1)
    lx, ly, lz = ((m * t).sum() for t in torch.linalg.cross(x.T, v.T).T)
    return torch.stack((0.5 * (m * (v * v).sum(0)).sum(), 0.5 * (m * phi).sum(), p[0], p[1], p[2], lx, ly, lz))


def exact(case, seed):
    """What run() returns on a fresh state, in 64 bits; None where that would take too long.  Positions keep the
    case's precision between the steps, as the caller's arrays do."""
    kind, n = case["kind"], case["n"]
    theta2 = case["theta"] ** 2
    x, v, m, off = (None,) * 4
    if kind == "direct":
        if n * case["targets"] > 2.0e10:
            return None
        x, v, m, off = _particles(case, seed)
        return _exact_direct(x, m, _targets(case, seed), case)
    if kind in ("ensemble", "grad") or n / theta2 > (6.0e6 if kind != "vjp" else 8.0e5):
        return None
    x, v, m, off = _particles(case, seed)
    if kind == "accel":
        return _exact_accel(x, m, case)
    if kind == "vjp":
        return _exact_vjp(x, m, *_cotangents(case, n, seed), case)
    a, _ = _exact_accel(x, m, case)
    tau, dt = case["tau"], _dtype(case)
    v1 = v.double() + 0.5 * tau * a
    x1 = (x.double() + tau * v1).to(dt)
    a1, phi = _exact_accel(x1, m, case)
    v1 = v1 + 0.5 * tau * a1
    return x1.double(), v1, a1, phi, _exact_diag(x1.double(), v1, m.double(), phi)
