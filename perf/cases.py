"""The work a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values; ``prepare`` makes what a program holds before the call (the grid
resident on the device, the rays or points of this pass, the buffers a loop of passes emits into), ``run`` is one pass through the package's
public entry points, ``work`` the bytes and operations no implementation can do without, and ``exact``
the results of the same pass from plain torch in 64 bits.

Sizes are those of the workloads in ``synth`` (the exponential disk at mass thresholds 1e-4 to 1e-6, the
clumpy ring torus of ~1e7 leaves, the uneven batch of grids) and of the tests (hundreds to thousands of
rays).  Rays are isotropic with origins uniform in the domain, or paths with both ends uniform in it;
weights are uniform and interaction depths exponential, as in the Monte Carlo loop.
"""
import math

import numpy as np
import torch

import paper_1311_0705_gb300 as hg
import synth

# ----------------------------------------------------------------------------- cases

DISK, TORUS = "disk", "torus"


def _case(name, path, n, tree="octree", model=DISK, delta=1e-6, level=12, **more):
    c = dict(name=name, path=path, n=n, tree=tree, model=model, delta=delta, level=level, nav="lists", precision="fp64",
             ends="free", kappa=1.0, grids=1)
    c.update(more)
    return c


def listed():
    return [
        # a handful of packets on a small grid: a scripted query, where launches and latency are all there is
        _case("trace_tiny", "trace", 255, delta=1e-4, level=6),
        # the plain workload: cell sequences and optical depths of 1e4 rays through ~1e4 leaves
        _case("emit_small", "emit", 10_000, delta=1e-4, level=6),
        # the main pass: optical depths of a new batch of emission rays on the large octree
        _case("trace_octree", "trace", 1_000_000),
        # one step of a radiative-transfer loop on the k-d tree: depths, emitted sequences and adjoint
        _case("step_kd", "step", 1_000_000, tree="kd"),
        # the largest grid and batch, in the reduced-precision mode offered for it
        _case("trace_torus_fp32k", "trace", 10_000_000, tree="kd", model=TORUS, delta=7e-7, level=10, precision="fp32k"),
        # packets walked to their next interaction point, in a medium of which a part interacts
        _case("interact_octree", "interact", 1_000_000, kappa=200.0),
        # grid quality: density at random points against the model
        _case("quality_rho_kd", "rho", 1_000_000, tree="kd"),
        # grid quality: optical depth along random paths against adaptive quadrature of the model
        _case("quality_tau_octree", "tau", 100_000, delta=1e-5, ends="both"),
        # many uneven grids in one launch (parameter studies)
        _case("batch_fp32k", "batch", 4_000_000, delta=1e-5, level=10, precision="fp32k", grids=12),
        # fitting leaf densities to optical depths along bounded paths: forward and backward through autograd
        _case("fit_kd", "fit", 300_007, tree="kd", delta=1e-5, ends="both"),
        # a mid-size octree walked by ropes, ragged ray count
        _case("trace_ropes", "trace", 200_003, delta=1e-5, nav="ropes"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    path = rng.choice(["trace", "trace", "trace", "emit", "step", "step", "interact", "rho", "tau", "batch", "fit"])
    c = _case("", path, int(_log(rng, 200, 2_000_000)), tree=rng.choice(["octree", "kd"]),
              delta=float("%.3g" % _log(rng, 1e-6, 1e-3)), level=rng.randint(6, 12))
    del c["name"]
    if path in ("trace", "emit", "step"):
        c["precision"] = rng.choice(["fp64", "fp64", "fp32k"])
        c["nav"] = rng.choice(["lists", "lists", "lists", "ropes"])
        c["ends"] = rng.choice(["free", "free", "both"])
        if c["tree"] == "kd" and rng.random() < 0.3:
            c["model"], c["delta"], c["level"] = TORUS, float("%.3g" % _log(rng, 5e-6, 1e-4)), rng.randint(6, 9)
    if path == "interact":
        c["kappa"] = float("%.3g" % _log(rng, 1.0, 1e3))
    if path in ("tau", "fit"):
        c["ends"], c["n"] = "both", int(_log(rng, 200, 300_000))
        c["delta"] = float("%.3g" % _log(rng, 3e-6, 1e-3))
    if path == "batch":
        c["grids"], c["precision"] = rng.randint(2, 20), rng.choice(["fp64", "fp32k"])
        c["n"], c["delta"], c["level"] = int(_log(rng, 20_000, 4_000_000)), float("%.3g" % _log(rng, 1e-5, 1e-3)), 10
    return c


# ----------------------------------------------------------------------------- inputs

KIND = {"octree": synth.TREE_OCTREE, "kd": synth.TREE_KD}


def _model(case):
    return synth.make_torus(synth.config_seed(3)) if case["model"] == TORUS else synth.make_disk()


def _params(case, i=0, kind=None, delta=None):
    p = synth.BuildParams(kind=KIND[case["tree"]] if kind is None else kind, delta_max=case["delta"] if delta is None else delta,
                          max_level=case["level"], seed=synth.config_seed(2) + i)
    if case["model"] == TORUS:
        p.use_tau, p.tau_max, p.use_q, p.q_max = True, 0.5, True, 0.9
    return p


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _rays(g, n, ends):
    """Origins uniform in the domain with isotropic directions, or paths between two uniform points."""
    o = 2.0 * _rand(g, n, 3) - 1.0
    if ends == "both":
        v = 2.0 * _rand(g, n, 3) - 1.0 - o
        length = v.square().sum(1).sqrt()
        return o, v / length[:, None], length
    mu, phi = 2.0 * _rand(g, n) - 1.0, 2.0 * math.pi * _rand(g, n)
    s = (1.0 - mu * mu).clamp_min(0.0).sqrt()
    return o, torch.stack([s * phi.cos(), s * phi.sin(), mu], 1), None


def _batch_plan(case):
    """Trees, thresholds and ray counts of a batch: uneven over a factor of ten and of thirty."""
    rng = np.random.default_rng(synth.config_seed(4) + case["grids"])
    kinds = rng.integers(0, 2, case["grids"])
    deltas = case["delta"] * 10.0 ** rng.uniform(0.0, 1.0, case["grids"])
    share = 30.0 ** rng.uniform(0.0, 1.0, case["grids"])
    cuts = np.floor(np.cumsum(share) / share.sum() * case["n"]).astype(np.int64)
    cuts[-1] = case["n"]
    return kinds, deltas, np.concatenate([[0], cuts])


def _capacity(case):
    """Entries a program sets aside for the emitted cells of a pass."""
    return int(1.6 * case["n"] * _crossings(case, _leaves(case))) + 4000


def prepare(case, seed):
    g = _generator(seed)
    path, n = case["path"], case["n"]
    model = _model(case)
    s = dict(case=case)
    host = None
    if path == "batch":
        kinds, deltas, begin = _batch_plan(case)
        s["grids"] = [hg.load_grid(hg.build_grid_gpu(model, _params(case, i, int(k), float(d))), validate=False)
                      for i, (k, d) in enumerate(zip(kinds, deltas))]
        s["batch"] = hg.Batch(s["grids"], begin)
    else:
        host = hg.build_grid_gpu(model, _params(case))
        s["grid"] = hg.load_grid(host, validate=False, nav=case["nav"])
    if path in ("rho", "tau"):
        s["dmodel"] = hg.load_model(model)
    if path == "rho":
        s["pts"] = 2.0 * _rand(g, n, 3) - 1.0
        return s
    s["o"], s["d"], s["s_max"] = _rays(g, n, case["ends"])
    if path == "step":
        s["w"] = _rand(g, n).float()
    if path in ("emit", "step"):
        real = torch.float32 if case["precision"] == "fp32k" else torch.float64
        s["emitted"] = (torch.zeros(_capacity(case), dtype=torch.int32, device="cuda"),
                        torch.zeros(_capacity(case), dtype=real, device="cuda"))
    if path == "interact":
        s["tau_int"] = -(1.0 - _rand(g, n)).log()
    if path == "fit":
        s["rho"] = torch.from_numpy(np.ascontiguousarray(host.leaf_rho)).cuda().requires_grad_()
        s["g_tau"] = _rand(g, n)
    return s


# ----------------------------------------------------------------------------- one pass

def run(s):
    c = s["case"]
    path = c["path"]
    if path == "trace":
        return hg.trace_rays(s["grid"], s["o"], s["d"], s["s_max"], kappa=c["kappa"], precision=c["precision"])
    if path == "emit":
        rays = hg.prepare_rays(s["grid"], s["o"], s["d"], s["s_max"])
        tau, ncross, status = rays.trace(kappa=c["kappa"], precision=c["precision"])
        off = hg.scan_offsets(ncross)
        cell, ds = rays.fill(off, precision=c["precision"], capacity=s["emitted"][0].shape[0], status=status, out=s["emitted"])
        rays.free()
        return tau, ncross, status, off, cell, ds
    if path == "step":
        rays = hg.prepare_rays(s["grid"], s["o"], s["d"], s["s_max"])
        tau, ncross, status, _ = rays.trace_stage(kappa=c["kappa"], precision=c["precision"])
        off = hg.scan_offsets(ncross)
        cell, ds, grad = rays.emit_staged_gradient(off, s["w"], kappa=c["kappa"], capacity=s["emitted"][0].shape[0],
                                                   status=status, out=s["emitted"])
        rays.free()
        return tau, ncross, status, off, cell, ds, grad
    if path == "interact":
        return hg.find_interactions(s["grid"], s["o"], s["d"], s["tau_int"], s["s_max"], kappa=c["kappa"])
    if path == "rho":
        cell, rho_g = hg.sample_density(s["grid"], s["pts"])
        rho_t = hg.model_density(s["dmodel"], s["pts"])
        return cell, rho_g, rho_t, hg.diff_stats(rho_t, rho_g)
    if path == "tau":
        tau_g, ncross, _ = hg.trace_rays(s["grid"], s["o"], s["d"], s["s_max"], kappa=c["kappa"])
        tau_t = hg.model_tau(s["dmodel"], s["o"], s["d"], s["s_max"], kappa=c["kappa"])
        return tau_g, ncross, tau_t, hg.diff_stats(tau_t, tau_g)
    if path == "batch":
        return s["batch"].trace(s["o"], s["d"], s["s_max"], kappa=c["kappa"], precision=c["precision"])
    if path == "fit":
        s["rho"].grad = None
        tau = hg.TauFn.apply(s["rho"], s["grid"], s["o"], s["d"], s["s_max"], c["kappa"])
        tau.backward(s["g_tau"])
        return tau.detach(), s["rho"].grad
    raise ValueError(path)


# ----------------------------------------------------------------------------- what a pass cannot do without

def _leaves(case, delta=None):
    """Leaves of the grids these thresholds give (the mass criterion halves a node until it holds delta)."""
    d = case["delta"] if delta is None else delta
    if case["model"] == TORUS:
        return min(6.9 / d, 0.07 * 8.0 ** case["level"])
    return min((3.35 if case["tree"] == "octree" else 1.45) / d, 0.05 * 8.0 ** case["level"] + 2000)


def _crossings(case, leaves):
    """Mean leaves crossed per ray: 30.9 and 25.5 on the disk grids of 3.35e6 and 1.45e6 leaves, 37.4 on the
    torus of 9.8e6, falling with about the 0.23th power of the leaf count (9.2 at 1.8e4 leaves)."""
    m = 37.4 * (leaves / 9.8e6) ** 0.23 if case["model"] == TORUS else 30.9 * (leaves / 3.35e6) ** 0.23
    if case["path"] == "interact":
        m *= 0.6
    return m * (0.9 if case["ends"] == "both" else 1.0)


def work(case):
    path, n = case["path"], case["n"]
    leaves = _leaves(case)
    if path == "rho":
        # in: points and the leaves' boxes and densities; out: cell, both densities, statistics
        return {"bytes": n * (24 + 4 + 16.0) + 56.0 * min(leaves, n), "flops": n * 40.0}
    if path == "batch":
        _, deltas, begin = _batch_plan(case)
        share = np.diff(begin)
        cross = sum(float(k) * _crossings(case, _leaves(case, float(d))) for k, d in zip(share, deltas))
        leaves = sum(_leaves(case, float(d)) for d in deltas)
    else:
        cross = n * _crossings(case, leaves)
    real = 4.0 if case["precision"] == "fp32k" else 8.0
    # in: origins, directions (and path ends), and once each leaf that is crossed: six bounds, density, wall
    # ranges and next leaf (76 bytes); out: depth, count, status
    b = n * (48.0 + (8.0 if case["ends"] == "both" else 0.0) + real + 5.0) + 76.0 * min(leaves, cross)
    f = 16.0 * cross  # three wall times, the exit point, the length, the sum
    if path == "emit":
        b += cross * (4.0 + real) + 8.0 * n
    if path == "step":
        b += cross * (4.0 + real) + 12.0 * n + 4.0 * leaves
        f += 2.0 * cross
    if path == "interact":
        b += 16.0 * n
    if path == "tau":
        b += 8.0 * n
        f += n * 600 * 30.0
    if path == "fit":
        b += 8.0 * n + 16.0 * leaves
        f += 2.0 * cross
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- the same in 64 bits, in plain torch

class _Tree:
    """A built grid's node list as torch arrays, with the split planes read off the children's boxes."""

    def __init__(self, host):
        up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        self.octree = host.kind == synth.TREE_OCTREE
        lo, hi = up(host.node_lo), up(host.node_hi)
        self.child, self.leaf = up(host.child_first).long(), up(host.node_leaf).long()
        first = self.child.clamp_min(0)
        self.split = hi[first]
        self.axis = (self.split != hi).long().argmax(1)
        node = torch.nonzero(self.leaf >= 0)[:, 0]
        self.lo, self.hi, self.rho = lo[node], hi[node], up(host.leaf_rho)
        self.dlo, self.dhi = lo[0], hi[0]

    def locate(self, p, d):
        """Leaf of each point; a point on a split plane belongs to the side its direction points to."""
        out = torch.empty(p.shape[0], dtype=torch.long, device=p.device)
        idx, nd = torch.arange(p.shape[0], device=p.device), torch.zeros(p.shape[0], dtype=torch.long, device=p.device)
        while idx.numel():
            c = self.child[nd]
            done = c < 0
            if bool(done.any()):
                out[idx[done]] = self.leaf[nd[done]]
                keep = ~done
                idx, nd, c = idx[keep], nd[keep], c[keep]
                if not idx.numel():
                    break
            up = (p[idx] > self.split[nd]) | ((p[idx] == self.split[nd]) & (d[idx] >= 0))
            if self.octree:
                nd = c + up[:, 0].long() + 2 * up[:, 1].long() + 4 * up[:, 2].long()
            else:
                nd = c + up.gather(1, self.axis[nd][:, None])[:, 0].long()
        return out


def _walk64(t, o, d, s_max, kappa=1.0, tau_int=None, emit=False):
    """Every path leaf by leaf: exit wall, exit point, next leaf from the root."""
    n = o.shape[0]
    S = torch.zeros(n, dtype=torch.float64, device="cuda")
    it = torch.zeros(n, dtype=torch.float64, device="cuda")
    act = torch.arange(n, device="cuda")
    cell, tc = t.locate(o, d), torch.zeros(n, dtype=torch.float64, device="cuda")
    segs = []
    ar3 = torch.arange(3, device="cuda")
    while act.numel():
        oo, dd, lo, hi = o[act], d[act], t.lo[cell], t.hi[cell]
        wall = torch.where(dd > 0, hi, lo)
        tw = torch.where(dd == 0, math.inf, (wall - oo) * (1.0 / dd))
        te, ax = tw.min(1)
        end = torch.zeros_like(act, dtype=torch.bool)
        if s_max is not None:
            end = s_max[act] < te
            te = torch.where(end, s_max[act], te)
        te = torch.maximum(te, tc)
        ds = te - tc
        Sn = S[act] + t.rho[cell] * ds
        stop = torch.zeros_like(end)
        if tau_int is not None:
            ti = tau_int[act]
            stop = (ds > 0) & (kappa * Sn >= ti)
            a, b = ti - kappa * S[act], kappa * t.rho[cell]
            at = torch.minimum(torch.where((a > 0) & (b > 0), tc + a / b, tc), te)
            it[act[stop]] = at[stop]
        S[act] = Sn
        if emit:
            r = ds > 0
            segs.append((act[r], cell[r], ds[r]))
        p = torch.minimum(torch.maximum(oo + dd * te[:, None], lo), hi)
        on = ar3[None, :] == ax[:, None]
        p = torch.where(on, wall, p)
        out = ((wall == torch.where(dd > 0, t.dhi, t.dlo)) & on).any(1)
        out |= (((p == t.dhi) & (dd > 0)) | ((p == t.dlo) & (dd < 0))).any(1)
        over = end | stop | out
        it[act[over & ~stop]] = te[over & ~stop]
        keep = ~over
        act, tc = act[keep], te[keep]
        if act.numel():
            cell = t.locate(p[keep], dd[keep])
    if emit:
        r, c, l = (torch.cat(x) for x in zip(*segs))
        order = torch.sort(r, stable=True).indices
        segs = (r[order], c[order], l[order])
    return S, it, segs


def _disk64(m, p):
    """Density of the exponential disk."""
    return m.params[0] * torch.exp(-(p[..., :2].square().sum(-1).sqrt() / m.params[1]) - p[..., 2].abs() / m.params[2])


def _disk_tau64(m, o, d, length):
    """Optical depth through the disk: the path cut at the midplane and at its closest approach to the axis,
    each piece integrated by Gauss-Legendre panels that shrink geometrically towards its ends."""
    x, wt = np.polynomial.legendre.leggauss(16)
    x, wt = torch.from_numpy(x).cuda(), torch.from_numpy(wt).cuda()
    cut = torch.stack([-o[:, 2] / d[:, 2], -(o[:, :2] * d[:, :2]).sum(1) / d[:, :2].square().sum(1)], 1)
    cut = torch.minimum(torch.nan_to_num(cut, nan=0.0).clamp_min(0.0), length[:, None]).sort(1).values
    edge = torch.cat([torch.zeros_like(length)[:, None], cut, length[:, None]], 1)
    f = [0.0] + [2.0 ** -k for k in range(30, 0, -1)]
    f = f + [1.0 - v for v in reversed(f[:-1])]
    tau = torch.zeros_like(length)
    for k in range(3):
        a, w = edge[:, k], edge[:, k + 1] - edge[:, k]
        for u0, u1 in zip(f[:-1], f[1:]):
            h = 0.5 * (u1 - u0) * w
            t = (a + 0.5 * (u0 + u1) * w)[:, None] + h[:, None] * x
            tau += h * (_disk64(m, o[:, None, :] + d[:, None, :] * t[..., None]) * wt).sum(1)
    return tau


def _stats64(a, b):
    x = a - b
    return torch.stack([torch.tensor(float(x.numel()), dtype=torch.float64, device="cuda"), x.mean(),
                        (x - x.mean()).square().mean().sqrt()])


def exact(case, seed):
    path, kappa, n = case["path"], case["kappa"], case["n"]
    model, g = _model(case), _generator(seed)
    if path == "rho":
        t, p = _Tree(hg.build_grid_gpu(model, _params(case))), 2.0 * _rand(g, n, 3) - 1.0
        rho_g, rho_t = t.rho[t.locate(p, torch.zeros_like(p))], _disk64(model, p)
        return None, rho_g, rho_t, _stats64(rho_t, rho_g)
    o, d, s_max = _rays(g, n, case["ends"])
    if path == "batch":
        kinds, deltas, begin = _batch_plan(case)
        tau = torch.empty(n, dtype=torch.float64, device="cuda")
        for i, (k, dl) in enumerate(zip(kinds, deltas)):
            t, r = _Tree(hg.build_grid_gpu(model, _params(case, i, int(k), float(dl)))), slice(int(begin[i]), int(begin[i + 1]))
            tau[r] = kappa * _walk64(t, o[r], d[r], None)[0]
        return tau, None, None
    t = _Tree(hg.build_grid_gpu(model, _params(case)))
    if path == "trace":
        return kappa * _walk64(t, o, d, s_max)[0], None, None
    if path in ("emit", "step"):
        w = _rand(g, n).float().double() if path == "step" else None
        S, _, (r, c, l) = _walk64(t, o, d, s_max, emit=True)
        ds = torch.zeros(_capacity(case), dtype=torch.float64, device="cuda")
        m = min(ds.numel(), l.numel())
        ds[:m] = l[:m]
        out = (kappa * S, None, None, None, None, ds)
        return out if w is None else out + (torch.zeros_like(t.rho).index_add_(0, c, kappa * w[r] * l),)
    if path == "interact":
        return None, _walk64(t, o, d, s_max, kappa=kappa, tau_int=-(1.0 - _rand(g, n)).log())[1], None, None
    if path == "tau":
        tau_g, tau_t = kappa * _walk64(t, o, d, s_max)[0], kappa * _disk_tau64(model, o, d, s_max)
        return tau_g, None, tau_t, _stats64(tau_t, tau_g)
    if path == "fit":
        g_tau = _rand(g, n)
        S, _, (r, c, l) = _walk64(t, o, d, s_max, emit=True)
        return kappa * S, torch.zeros_like(t.rho).index_add_(0, c, kappa * g_tau[r] * l)
    raise ValueError(path)
