"""Performance cases: the calls a user of the solver makes, over the range of
meshes, degrees, precisions and options it is used with.

A case is a dict of plain values.  Its ``kind`` says which call one pass makes:

* ``vcycle``: ``Multigrid.vcycle``, the preconditioner applied inside a user's
  own Krylov method (one call per iteration, the handle kept);
* ``solve``: ``Multigrid.solve``, FGMRES to a relative residual;
* ``field``: a new coefficient field from set-up to solution (hierarchy, load
  vector, solve), as parameter studies and data generation run it;
* ``batch``: ``Batch.vcycle``, independent problems with several right-hand
  sides each;
* ``residual``: ``Multigrid.residual_norm`` with the residual vector, the
  operator's own cost (FP64, as the outer solver evaluates it);
* ``gradients``: ``CNN.gradients``, one backward pass of the learned initial
  guess on a minibatch.

Results that were computed in FP32 are returned as FP32, whatever type the call
hands them back in.
"""
import math

import numpy as np
import torch

from paper_1602_04858_gb300 import inputs, mgdarcy

DEV = "cuda"


def listed():
    return [
        # the smallest hierarchy in use (16^2 RT_0, one smoothing step, standard cycle): launches and latency
        dict(name="vcycle_16_rt0_fp64", kind="vcycle", dim=2, n_coarse=2, levels=4, degree=0, mu=1.0,
             precision="fp64", m_fine=1, variable=False, field="lognormal", sigma=1.0, nrhs=1),
        # the benchmark: channelised permeability at contrast 1e6, variable cycle, mixed precision
        dict(name="vcycle_channels_256_rt1_fp32", kind="vcycle", dim=2, n_coarse=4, levels=7, degree=1, mu=0.01,
             precision="fp32", m_fine=2, variable=True, field="channels", sigma=0.0, nrhs=1),
        # the same mesh in the paper's own precision
        dict(name="vcycle_channels_256_rt1_fp64", kind="vcycle", dim=2, n_coarse=4, levels=7, degree=1, mu=0.01,
             precision="fp64", m_fine=2, variable=True, field="channels", sigma=0.0, nrhs=1),
        # a mesh that is no power of two, BF16 patch inverses, the standard V(2,2) cycle
        dict(name="vcycle_192_rt1_bf16inv_v22", kind="vcycle", dim=2, n_coarse=3, levels=7, degree=1, mu=0.01,
             precision="fp32_bf16inv", m_fine=2, variable=False, field="lognormal", sigma=2.0, nrhs=1),
        # 3-D Darcy flow in a lognormal field
        dict(name="vcycle_3d_64_rt0_fp32", kind="vcycle", dim=3, n_coarse=2, levels=6, degree=0, mu=0.0,
             precision="fp32", m_fine=2, variable=True, field="lognormal", sigma=3.0, nrhs=1),
        # the highest degree: 96-dof patches
        dict(name="vcycle_128_rt2_fp32", kind="vcycle", dim=2, n_coarse=4, levels=6, degree=2, mu=0.01,
             precision="fp32", m_fine=2, variable=True, field="channels", sigma=0.0, nrhs=1),
        # independent problems of two sizes, four right-hand sides each
        dict(name="batch_64_128_rt1_fp32", kind="batch", dim=2, n_coarse=4, levels=6, problems=2, degree=1, mu=0.01,
             precision="fp32", m_fine=2, variable=True, field="lognormal", sigma=2.0, nrhs=4),
        # time to a 1e-8 residual on the benchmark problem, mixed precision
        dict(name="solve_channels_256_rt1_fp32", kind="solve", dim=2, n_coarse=4, levels=7, degree=1, mu=0.01,
             precision="fp32", m_fine=2, variable=True, field="channels", sigma=0.0, nrhs=1, tol=1e-8),
        # a 3-D Brinkman solve in FP64 on a mesh that is no power of two
        dict(name="solve_3d_24_rt0_fp64", kind="solve", dim=3, n_coarse=3, levels=4, degree=0, mu=0.01,
             precision="fp64", m_fine=2, variable=True, field="lognormal", sigma=2.0, nrhs=1, tol=1e-8),
        # one sample of a parameter study: a new 128^2 field set up and solved
        dict(name="field_128_rt0_fp32", kind="field", dim=2, n_coarse=4, levels=6, degree=0, mu=0.01,
             precision="fp32", m_fine=2, variable=True, field="lognormal", sigma=2.0, nrhs=1, tol=1e-10),
        # the FP64 residual of a large level
        dict(name="residual_320_rt1_fp64", kind="residual", dim=2, n_coarse=5, levels=7, degree=1, mu=0.01,
             precision="fp32", m_fine=2, variable=True, field="lognormal", sigma=2.0, nrhs=1),
        # gradients of the learned guess on a minibatch of 128^2 fields
        dict(name="gradients_16x128", kind="gradients", n=128, batch=16),
    ]


def draw(rng):
    kind = rng.choice(["vcycle"] * 6 + ["solve", "field", "batch", "residual", "gradients"])
    if kind == "gradients":
        return dict(kind=kind, n=int(round(math.exp(rng.uniform(math.log(24), math.log(128))))),
                    batch=rng.randint(1, 16))
    dim = 3 if kind in ("vcycle", "solve") and rng.random() < 0.25 else 2
    degree = 0 if dim == 3 or kind == "field" else rng.choice([0, 1, 1, 2] if kind in ("vcycle", "residual") else [0, 1])
    top = {(3, 0): 64, (2, 0): 384, (2, 1): 256, (2, 2): 128}[dim, degree]
    if kind != "vcycle":
        top = {"solve": 40 if dim == 3 else 160, "field": 128, "batch": 128, "residual": top}[kind]
    n = math.exp(rng.uniform(math.log(8 if dim == 3 else 16), math.log(top)))
    n_coarse = rng.randint(2, 4 if dim == 3 else 7)
    levels = max(3, int(round(math.log2(n / n_coarse))) + 1)
    while (n_coarse << (levels - 1)) > top:
        levels -= 1
    precision = rng.choice(["fp32", "fp32", "fp64", "fp32_bf16inv"])
    if kind in ("field", "batch"):
        precision = "fp32"
    field = "lognormal"
    if dim == 2 and (kind == "vcycle" or (kind == "solve" and precision != "fp64")) and rng.random() < 0.3:
        field = "channels"
    mu = 0.01 if field == "channels" else rng.choice([0.0, 0.01, 0.01, 1.0])
    case = dict(kind=kind, dim=dim, n_coarse=n_coarse, levels=levels, degree=degree, mu=mu,
                precision=precision, m_fine=rng.choice([1, 2, 2]), variable=rng.random() < 0.7, field=field,
                sigma=round(rng.uniform(1.0, 2.0), 2), nrhs=1)
    if kind == "vcycle" and degree < 2 and rng.random() < 0.25:
        case["nrhs"] = rng.randint(2, 5)
    if kind == "batch":
        case.update(nrhs=rng.randint(1, 5), problems=rng.randint(2, 3))
    if kind in ("solve", "field"):
        case["tol"] = 1e-8
    return case


# --- inputs ------------------------------------------------------------------

def _n(case):
    return case["n_coarse"] << (case["levels"] - 1)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _grf(gen, n, d, sigma, ell):
    """Gaussian random field with covariance sigma^2 exp(-r^2 / (2 ell^2)), r in cells."""
    m = n + int(4 * ell)
    w = torch.randn((m,) * d, generator=gen, dtype=torch.float64, device=DEV)
    r = torch.arange(m, dtype=torch.float64, device=DEV)
    r = torch.minimum(r, m - r)
    cov = torch.full((m,) * d, sigma * sigma, dtype=torch.float64, device=DEV)
    for e in range(d):
        cov = cov * torch.exp(-r * r / (2 * ell * ell)).reshape([-1 if f == e else 1 for f in range(d)])
    spec = torch.fft.fftn(cov).real.clamp_min(0.0)
    g = torch.fft.ifftn(spec.sqrt() * torch.fft.fftn(w)).real
    return g[(slice(0, n),) * d].contiguous()


def _field(case, seed, n):
    """Zero-order coefficient c, one value per cell (axis order z, y, x)."""
    if case["field"] == "channels":
        return torch.as_tensor(inputs.channel_c(n, 20, seed), device=DEV)
    return torch.exp(_grf(_gen(seed), n, case["dim"], case["sigma"], max(1.0, n / 16)))


def _sizes(d, k, n):
    N = n * (k + 1)
    return d * (N + 1) * N ** (d - 1), N ** d


def _constrained(d, k, n):
    N = n * (k + 1)
    out = []
    for i in range(d):
        m = torch.zeros([N + 1 if d - 1 - a == i else N for a in range(d)], dtype=torch.bool, device=DEV)
        m.select(d - 1 - i, 0).fill_(True)
        m.select(d - 1 - i, N).fill_(True)
        out.append(m.reshape(-1))
    return torch.cat(out + [torch.zeros(N ** d, dtype=torch.bool, device=DEV)])


def _vectors(case, seed, n, count):
    """Random vectors, zero on the constrained dofs: residuals with a compatible
    pressure block, or loads without a divergence source for a solve."""
    nu, npr = _sizes(case["dim"], case["degree"], n)
    r = torch.randn((count, nu + npr), generator=_gen(seed + 7), dtype=torch.float64, device=DEV)
    if case["kind"] == "solve":
        r[:, nu:] = 0.0
    else:
        r[:, nu:] -= r[:, nu:].mean(dim=1, keepdim=True)
    r[:, _constrained(case["dim"], case["degree"], n)] = 0.0
    return r


def _args(case, c):
    return dict(dim=case["dim"], n_coarse=case["n_coarse"], n_levels=case["levels"], degree=case["degree"],
                mu=case["mu"], c=c, precision=case["precision"], m_fine=case["m_fine"],
                variable_cycle=case["variable"])


def _batch_levels(case):
    """Level counts of a batch's problems: the largest mesh and the next coarser one, alternating."""
    return [case["levels"] - (p % 2) for p in range(2 * case["problems"])]


def _params(seed):
    rng = np.random.default_rng(seed)
    out = []
    for ci, co in ((3, 32), (32, 32), (32, 32), (32, 3)):
        out += [rng.standard_normal(co * ci * 9) * math.sqrt(2.0 / (9 * ci)), 0.1 * rng.standard_normal(co)]
    return np.concatenate(out).astype(np.float32)


def _images(case, seed):
    """Normalised features and smooth targets of a minibatch (batch x 3 x n x n)."""
    gen = _gen(seed)
    n, b = case["n"], case["batch"]
    x = torch.stack([torch.stack([_grf(gen, n, 2, 1.0, n / 16), _grf(gen, n, 2, 1.0, n / 8), _grf(gen, n, 2, 1.0, n / 8)])
                     for _ in range(b)])
    y = torch.stack([torch.stack([_grf(gen, n, 2, 1.0, n / 8) for _ in range(3)]) for _ in range(b)])
    return x.float().contiguous(), y.float().contiguous()


def prepare(case, seed):
    if case["kind"] == "gradients":
        net = mgdarcy.CNN(case["n"], max_batch=case["batch"], seed=0)
        net.set_params(_params(seed))
        x, y = _images(case, seed)
        return dict(case=case, net=net, x=x, y=y)
    n = _n(case)
    if case["kind"] == "batch":
        probs, r = [], []
        for p, lev in enumerate(_batch_levels(case)):
            sub = dict(case, levels=lev)
            probs.append(_args(sub, _field(sub, seed + 101 * p, _n(sub))))
            r.append(_vectors(sub, seed + 101 * p, _n(sub), case["nrhs"]).reshape(-1))
        r = torch.cat(r)
        return dict(case=case, B=mgdarcy.Batch(probs, nrhs=case["nrhs"]), r=r, z=torch.zeros_like(r))
    c = _field(case, seed, n)
    if case["kind"] == "field":
        gen = _gen(seed + 3)
        f = torch.stack([_grf(gen, n, 2, 1.0, n / 8) for _ in range(2)]).reshape(-1).contiguous()
        return dict(case=case, c=c, f=f)
    r = _vectors(case, seed, n, case["nrhs"])
    if case["kind"] == "residual":
        # a user of the operator alone: no dense fold
        G = mgdarcy.Multigrid(**_args(case, c), dense_level=0)
        x = torch.randn(r.numel(), generator=_gen(seed + 9), dtype=torch.float64, device=DEV)
        return dict(case=case, G=G, x=x, b=r.reshape(-1), r=torch.zeros_like(x))
    G = mgdarcy.Multigrid(**_args(case, c), nrhs=case["nrhs"])
    if case["kind"] == "solve":
        nu, _ = _sizes(case["dim"], case["degree"], n)
        r = r.reshape(-1)
        return dict(case=case, G=G, f=r[:nu].contiguous(), g=r[nu:].contiguous(), x=torch.zeros_like(r))
    r = r.reshape(-1)
    return dict(case=case, G=G, r=r, z=torch.zeros_like(r))


def _result(case, z):
    return z if case["precision"] == "fp64" else z.to(torch.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "vcycle":
        state["G"].vcycle(state["r"], state["z"])
        return _result(case, state["z"])
    if kind == "batch":
        state["B"].vcycle(state["r"], state["z"])
        return _result(case, state["z"])
    if kind == "solve":
        state["G"].solve(state["f"], state["g"], state["x"], tol=case["tol"], maxit=300, check=False)
        return _result(case, state["x"])
    if kind == "field":
        n = _n(case)
        G = mgdarcy.Multigrid(**_args(case, state["c"]), dense_level=max(0, case["levels"] - 4))
        nu, npr = _sizes(2, case["degree"], n)
        b = torch.zeros(nu + npr, dtype=torch.float64, device=DEV)
        G.load_vector(state["f"], None, b)
        x = torch.zeros_like(b)
        G.solve(b[:nu].contiguous(), b[nu:].contiguous(), x, tol=case["tol"], maxit=400, check=False)
        G.close()
        return b, _result(case, x)
    if kind == "residual":
        norm = state["G"].residual_norm(state["x"], state["b"], state["r"])
        return state["r"], norm
    loss, grads = state["net"].gradients(state["x"], state["y"], case["batch"])
    return loss, grads


# --- what a pass cannot do without ---------------------------------------------

def _row_nnz(d, k, mu):
    """Average nonzeros of a velocity row and of a pressure row, interior of the mesh."""
    own = ((2 * k + 3) + k * (k + 2)) / (k + 1)
    visc = 1 + (d - 1) * (3 * (k + 1) - 1) if mu > 0 else 1
    return own * visc + (k + 2), d * (k + 2)


def _cycle_work(d, k, mu, n_coarse, levels, m_fine, variable, nrhs, s_bytes):
    """One V-cycle: every patch inverse read once, r and z in FP64, the smoothing operations."""
    nu, npr = _sizes(d, k, n_coarse << (levels - 1))
    nbytes, flops = 16.0 * nrhs * (nu + npr), 0.0
    ru, rp = _row_nnz(d, k, mu)
    nvu, nvp = d * (2 * k + 1) * (2 * k + 2) ** (d - 1), (2 * k + 2) ** d
    nv = nvu + nvp
    for j in range(1, levels):
        patches = ((n_coarse << j) - 1) ** d
        m = m_fine * (2 ** (levels - 1 - j) if variable else 1)
        sweeps = 2 * m * (2 * 3 ** d - 1) / 3 ** d
        nbytes += patches * nv * nv * s_bytes
        flops += nrhs * sweeps * patches * 2.0 * (nvu * ru + nvp * rp + nv * nv)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "gradients":
        px = case["batch"] * case["n"] ** 2
        macs = 9 * (3 * 32 + 32 * 32 + 32 * 32 + 32 * 3)
        # forward, weight gradients, input gradients (not of the first layer)
        return {"bytes": 24.0 * px + 8.0 * (macs + 99), "flops": 2.0 * px * (3 * macs - 9 * 3 * 32)}
    d, k, n, mu = case["dim"], case["degree"], _n(case), case["mu"]
    nu, npr = _sizes(d, k, n)
    s_bytes = {"fp64": 8, "fp32": 4, "fp32_bf16inv": 2}[case["precision"]]
    cyc = (d, k, mu, case["n_coarse"])
    tail = (case["m_fine"], case["variable"], case["nrhs"], s_bytes)
    ru, rp = _row_nnz(d, k, mu)
    if kind == "vcycle":
        b, f = _cycle_work(*cyc, case["levels"], *tail)
    elif kind == "batch":
        parts = [_cycle_work(*cyc, lev, *tail) for lev in _batch_levels(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "residual":
        b, f = 24.0 * (nu + npr) + 8.0 * n ** d, 2.0 * (nu * ru + npr * rp)
    else:   # ten iterations, the order of magnitude of a solve
        b, f = _cycle_work(*cyc, case["levels"], *tail)
        b, f = 10 * b, 10 * (f + 2.0 * (nu * ru + npr * rp))
        if kind == "field":
            nv = d * (2 * k + 1) * (2 * k + 2) ** (d - 1) + (2 * k + 2) ** d
            f += 2.0 * n ** d * (nv + 1) ** 3
    return {"bytes": b, "flops": f}


# --- plain 64-bit reference ------------------------------------------------------

def _lagrange(nodes, x):
    """Values and derivatives of the Lagrange basis through `nodes` at points x: (len(nodes), len(x))."""
    v = np.ones((len(nodes), len(x)))
    g = np.zeros((len(nodes), len(x)))
    for a, za in enumerate(nodes):
        for m, zm in enumerate(nodes):
            if m == a:
                continue
            g[a] = g[a] * (x - zm) / (za - zm) + v[a] / (za - zm)
            v[a] = v[a] * (x - zm) / (za - zm)
    return v, g


class _Ref1D:
    """1-D matrices of the nodal basis on [0, 1], unit cell size."""

    def __init__(self, k):
        t, w = np.polynomial.legendre.leggauss(k + 1)
        self.g, self.wg = (t + 1) / 2, w / 2
        c = np.zeros(k + 2)
        c[-1] = 1.0
        inner = np.sort(np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c)).real)
        self.gl = (np.concatenate(([-1.0], inner, [1.0])) + 1) / 2
        t, w = np.polynomial.legendre.leggauss(k + 2)
        t, w = (t + 1) / 2, w / 2
        lv, lg = _lagrange(self.gl, t)
        pv, pg = _lagrange(self.g, t)
        self.M, self.K = (lv * w) @ lv.T, (lg * w) @ lg.T
        self.Kd, self.G = (pg * w) @ pg.T, (pv * w) @ lg.T
        (v1, d1), (v0, d0) = _lagrange(self.g, np.ones(1)), _lagrange(self.g, np.zeros(1))
        s2 = 2.0 * (k + 1) * (k + 2)
        self.F = {}
        for a, (va, da, sa) in enumerate(((v1, d1, 1.0), (v0, d0, -1.0))):
            for b, (vb, db, sb) in enumerate(((v1, d1, 1.0), (v0, d0, -1.0))):
                self.F[a, b] = s2 * sa * sb * va @ vb.T - 0.5 * sa * va @ db.T - 0.5 * sb * da @ vb.T
        self.Blo = s2 * v0 @ v0.T + v0 @ d0.T + d0 @ v0.T
        self.Bhi = s2 * v1 @ v1.T - v1 @ d1.T - d1 @ v1.T

    def own(self, local, n, k):
        """Global matrix along a component's own direction from a cell matrix (shared face nodes)."""
        K1 = k + 1
        A = np.zeros((n * K1 + 1, n * K1 + 1))
        for c in range(n):
            A[c * K1:c * K1 + K1 + 1, c * K1:c * K1 + K1 + 1] += local
        return A

    def across(self, n, k):
        """Interior-penalty operator across a component's direction."""
        K1 = k + 1
        A = np.zeros((n * K1, n * K1))
        for c in range(n):
            A[c * K1:c * K1 + K1, c * K1:c * K1 + K1] += self.Kd
            if c + 1 < n:
                sl = [slice(c * K1, c * K1 + K1), slice((c + 1) * K1, (c + 2) * K1)]
                for a in (0, 1):
                    for b in (0, 1):
                        A[sl[a], sl[b]] += self.F[a, b]
        A[:K1, :K1] += self.Blo
        A[-K1:, -K1:] += self.Bhi
        return A

    def div(self, n, k):
        K1 = k + 1
        A = np.zeros((n * K1, n * K1 + 1))
        for c in range(n):
            A[c * K1:c * K1 + K1, c * K1:c * K1 + K1 + 1] += self.G
        return A


def _kron(mats):
    """COO (row, col, value) of the Kronecker product; mats in order x, y, z (x fastest)."""
    row = col = torch.zeros(1, dtype=torch.int64, device=DEV)
    val = torch.ones(1, dtype=torch.float64, device=DEV)
    rs = cs = 1
    for m in mats:
        m = torch.as_tensor(m, device=DEV)
        i, j = torch.nonzero(m, as_tuple=True)
        row = (row[None, :] + i[:, None] * rs).reshape(-1)
        col = (col[None, :] + j[:, None] * cs).reshape(-1)
        val = (val[None, :] * m[i, j][:, None]).reshape(-1)
        rs, cs = rs * m.shape[0], cs * m.shape[1]
    return row, col, val


class _RefLevel:
    """Operator, patches and patch inverses of one level, assembled."""

    def __init__(self, d, k, n, mu, c, patches):
        self.d, self.k, self.n = d, k, n
        K1, N = k + 1, n * (k + 1)
        self.N = N
        T = _Ref1D(k)
        self.T = T
        h = 1.0 / n
        nu, npr = _sizes(d, k, n)
        self.nu, self.ndof = nu, nu + npr
        comp = nu // d
        wper = np.diag(np.tile(T.wg, n))
        rows, cols, vals = [], [], []

        def add(t, ro, co, scale):
            rows.append(t[0] + ro)
            cols.append(t[1] + co)
            vals.append(t[2] * scale)

        cm = _constrained(d, k, n)
        cc = c.reshape(-1)
        grids = torch.arange(n ** d, device=DEV)
        cell = [(grids // n ** e) % n for e in range(d)]
        for i in range(d):
            if mu != 0.0:
                for e in range(d):
                    mats = [T.own(T.K if e == i else T.M, n, k) if f == i else (T.across(n, k) if f == e else wper)
                            for f in range(d)]
                    add(_kron(mats), i * comp, i * comp, mu * h ** (d - 2))
            B = _kron([T.div(n, k) if f == i else wper for f in range(d)])
            add(B, nu, i * comp, -h ** (d - 1))
            add((B[1], B[0], B[2]), i * comp, nu, -h ** (d - 1))
            # cellwise coefficient: Gauss-Lobatto mass along x_i, Gauss weights across
            stride = [1] * d
            for f in range(1, d):
                stride[f] = stride[f - 1] * (N + 1 if f - 1 == i else N)
            for b in np.ndindex(*([K1] * (d - 1))):
                off = iter(b)
                base = torch.zeros_like(grids)
                wt = h ** d
                for f in range(d):
                    if f == i:
                        base = base + cell[f] * K1 * stride[f]
                    else:
                        q = next(off)
                        base = base + (cell[f] * K1 + q) * stride[f]
                        wt *= T.wg[q]
                for a in range(k + 2):
                    for ap in range(k + 2):
                        add((base + a * stride[i], base + ap * stride[i], cc * T.M[a, ap]), i * comp, i * comp, wt)
        r, q, v = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        keep = ~(cm[r] | cm[q])
        r, q, v = r[keep], q[keep], v[keep]
        ci = torch.nonzero(cm).reshape(-1)
        r, q, v = torch.cat([r, ci]), torch.cat([q, ci]), torch.cat([v, torch.ones_like(ci, dtype=torch.float64)])
        A = torch.sparse_coo_tensor(torch.stack([r, q]), v, (self.ndof, self.ndof)).coalesce()
        self.key = A.indices()[0] * self.ndof + A.indices()[1]
        self.val = A.values()
        self.A = A.to_sparse_csr()
        self.cm = cm
        w = torch.zeros(self.ndof, dtype=torch.float64, device=DEV)
        pw = torch.full((1,), h ** d, dtype=torch.float64, device=DEV)
        for _ in range(d):
            pw = (torch.as_tensor(np.tile(T.wg, n), device=DEV)[:, None] * pw[None, :]).reshape(-1)
        w[nu:] = pw
        self.w = w
        self.colours = self._patches() if patches else []

    def entries(self, dofs):
        """Dense A[dofs_p][:, dofs_p] of every row of `dofs`."""
        nv = dofs.shape[1]
        out = torch.zeros((dofs.shape[0], nv, nv), dtype=torch.float64, device=DEV)
        step = max(1, 40_000_000 // (nv * nv))
        for s in range(0, dofs.shape[0], step):
            dd = dofs[s:s + step]
            q = (dd[:, :, None] * self.ndof + dd[:, None, :]).reshape(-1)
            pos = torch.searchsorted(self.key, q).clamp_max(self.key.numel() - 1)
            out[s:s + step] = torch.where(self.key[pos] == q, self.val[pos], 0.0).reshape(dd.shape[0], nv, nv)
        return out

    def bordered_inverse(self, dofs):
        A = self.entries(dofs)
        P, nv = dofs.shape
        B = torch.zeros((P, nv + 1, nv + 1), dtype=torch.float64, device=DEV)
        B[:, :nv, :nv] = A
        B[:, :nv, nv] = B[:, nv, :nv] = self.w[dofs]
        return torch.cat([torch.linalg.inv(b)[:, :nv, :nv] for b in B.split(4096)])

    def _patches(self):
        d, K1, N, n = self.d, self.k + 1, self.N, self.n
        local = []
        for i in range(d + 1):
            dims = [N + 1 if f == i else N for f in range(d)]
            idx = torch.zeros(1, dtype=torch.int64, device=DEV)
            st = 1
            stride = []
            for f in range(d):
                r = torch.arange(2 * K1 - 1, device=DEV) + 1 if f == i else torch.arange(2 * K1, device=DEV)
                idx = (idx[None, :] + r[:, None] * st).reshape(-1)
                stride.append(st)
                st *= dims[f]
            local.append((idx + i * (self.nu // d), stride))
        out = []
        for col in range(3 ** d):
            v = [torch.arange((col // 3 ** e) % 3 or 3, n, 3, device=DEV) for e in range(d)]
            if any(x.numel() == 0 for x in v):
                out.append(None)
                continue
            vs = torch.stack([g.reshape(-1) for g in torch.meshgrid(*v, indexing="ij")])
            dofs = torch.cat([sum((vs[e] - 1) * K1 * st[e] for e in range(d))[:, None] + idx[None, :]
                              for idx, st in local], dim=1)
            out.append((dofs, self.bordered_inverse(dofs)))
        return out


class _Ref:
    """The V-cycle of the case in FP64, from its definition; vectors (ndof, right-hand sides)."""

    def __init__(self, case, c):
        d, k = case["dim"], case["degree"]
        self.case = case
        cs = [c]
        for _ in range(case["levels"] - 1):
            a = cs[-1]
            for e in range(d):
                a = a.unfold(e, 2, 2).mean(dim=-1)
            cs.append(a.contiguous())
        cs.reverse()
        self.lv = [_RefLevel(d, k, case["n_coarse"] << j, case["mu"], cs[j], j > 0) for j in range(case["levels"])]
        self.P = [None] + [self._prolong(j) for j in range(1, case["levels"])]
        self.Pt = [None] + [p.transpose(0, 1).to_sparse_csr() for p in self.P[1:]]
        self.P = [None] + [p.to_sparse_csr() for p in self.P[1:]]
        L0 = self.lv[0]
        self.free0 = torch.nonzero(~L0.cm).reshape(-1)
        self.inv0 = L0.bordered_inverse(self.free0[None, :])[0]

    def _prolong(self, j):
        d, k = self.case["dim"], self.case["degree"]
        K1, nc = k + 1, self.case["n_coarse"] << (j - 1)
        T = self.lv[0].T
        own = np.zeros((2 * nc * K1 + 1, nc * K1 + 1))
        per = np.zeros((2 * nc * K1, nc * K1))
        for f in range(2 * nc):
            c = f // 2
            own[f * K1:f * K1 + K1 + 1, c * K1:c * K1 + K1 + 1] = _lagrange(T.gl, (f % 2 + T.gl) / 2)[0].T
            per[f * K1:f * K1 + K1, c * K1:c * K1 + K1] = _lagrange(T.g, (f % 2 + T.g) / 2)[0].T
        Lf, Lc = self.lv[j], self.lv[j - 1]
        rows, cols, vals = [], [], []
        for i in range(d + 1):
            r, c, v = _kron([own if e == i else per for e in range(d)])
            rows.append(r + i * (Lf.nu // d))
            cols.append(c + i * (Lc.nu // d))
            vals.append(v)
        r, c, v = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        v = torch.where(Lf.cm[r] | Lc.cm[c], 0.0, v)
        return torch.sparse_coo_tensor(torch.stack([r, c]), v, (Lf.ndof, Lc.ndof)).coalesce()

    def level(self, j, b):
        L = self.lv[j]
        x = torch.zeros_like(b)
        if j == 0:
            x[self.free0] = self.inv0 @ b[self.free0]
            return x
        m = self.case["m_fine"] * (2 ** (len(self.lv) - 1 - j) if self.case["variable"] else 1)
        x = self._smooth(L, x, b, m)
        r = b - L.A @ x
        r[L.cm] = 0.0
        x = x + self.P[j] @ self.level(j - 1, self.Pt[j] @ r)
        return self._smooth(L, x, b, m)

    @staticmethod
    def _smooth(L, x, b, m):
        C = len(L.colours)
        for _ in range(m):
            for col in list(range(C)) + list(range(C - 2, -1, -1)):
                if L.colours[col] is not None:
                    dofs, S = L.colours[col]
                    x[dofs] += torch.bmm(S, (b - L.A @ x)[dofs])
        return x

    def vcycle(self, r):
        """r, z: (right-hand sides, ndof)."""
        cm = self.lv[-1].cm
        b = r.t().contiguous()
        b[cm] = 0.0
        z = self.level(len(self.lv) - 1, b)
        z[cm] = r.t()[cm]
        return z.t().contiguous()

    def solve(self, b, tol=1e-13, maxit=120):
        """Right-preconditioned flexible GMRES to a residual far below the case's own."""
        A = self.lv[-1].A
        V, Z, H = [b / b.norm()], [], torch.zeros((maxit + 1, maxit), dtype=torch.float64)
        for i in range(maxit):
            Z.append(self.vcycle(V[i][None, :])[0])
            w = A @ Z[i]
            for _ in range(2):
                B = torch.stack(V)
                h = B @ w
                w = w - B.t() @ h
                H[:i + 1, i] += h.cpu()
            H[i + 1, i] = float(w.norm())
            V.append(w / w.norm())
            e = torch.zeros(i + 2, dtype=torch.float64)
            e[0] = float(b.norm())
            y = torch.linalg.lstsq(H[:i + 2, :i + 1], e[:, None], driver="gelsd").solution[:, 0]
            if float((H[:i + 2, :i + 1] @ y - e).norm()) <= tol * float(b.norm()):
                break
        x = torch.stack(Z).t() @ y.to(DEV)
        L = self.lv[-1]
        x[L.nu:] -= (L.w @ x) / L.w.sum()
        return x


def _load(case, f):
    """Load vector of a cellwise-constant body force, from the integrals of the basis functions."""
    k, n = case["degree"], _n(case)
    T, K1, h = _Ref1D(k), case["degree"] + 1, 1.0 / _n(case)
    f = f.reshape(2, n, n)
    M = torch.as_tensor(T.M.sum(axis=1), device=DEV)
    wg = torch.as_tensor(T.wg, device=DEV)
    out = []
    for i in range(2):
        a = f[i] if i == 0 else f[i].t()          # own direction last
        u = torch.zeros((n * K1, n * K1 + 1), dtype=torch.float64, device=DEV)
        for q in range(k + 2):
            u[:, q:q + (n - 1) * K1 + 1:K1] += torch.kron(a, wg[:, None]) * M[q] * h * h
        u[:, 0] = u[:, -1] = 0.0
        out.append((u if i == 0 else u.t()).reshape(-1))
    return torch.cat(out + [torch.zeros((n * K1) ** 2, dtype=torch.float64, device=DEV)])


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradients":
        x, y = (t.double() for t in _images(case, seed))
        p = torch.as_tensor(_params(seed), device=DEV).double().requires_grad_(True)
        a, o = x, 0
        for l, (ci, co) in enumerate(((3, 32), (32, 32), (32, 32), (32, 3))):
            w = p[o:o + co * ci * 9].reshape(co, ci, 3, 3)
            bias = p[o + co * ci * 9:o + co * ci * 9 + co]
            o += co * ci * 9 + co
            # 3 x 3 convolution as a matrix product of the unfolded neighbourhoods
            u = torch.nn.functional.unfold(a if l == 0 else a.relu(), 3, padding=1)
            a = (w.reshape(co, -1) @ u).reshape(x.shape[0], co, case["n"], case["n"]) + bias[None, :, None, None]
        loss = ((a - y) ** 2).mean()
        loss.backward()
        return float(loss.detach()), p.grad.detach().cpu().numpy()
    n = _n(case)
    if kind == "batch":
        z = []
        for p, lev in enumerate(_batch_levels(case)):
            sub = dict(case, levels=lev)
            ref = _Ref(sub, _field(sub, seed + 101 * p, _n(sub)))
            z.append(ref.vcycle(_vectors(sub, seed + 101 * p, _n(sub), case["nrhs"])).reshape(-1))
        return torch.cat(z)
    c = _field(case, seed, n)
    if kind == "residual":
        L = _RefLevel(case["dim"], case["degree"], n, case["mu"], c, False)
        b = _vectors(case, seed, n, 1).reshape(-1)
        x = torch.randn(b.numel(), generator=_gen(seed + 9), dtype=torch.float64, device=DEV)
        r = b - L.A @ x
        return r, float(r.norm())
    if kind == "vcycle":
        return _Ref(case, c).vcycle(_vectors(case, seed, n, case["nrhs"])).reshape(-1)
    nu, npr = _sizes(case["dim"], case["degree"], n)
    if kind == "field":
        gen = _gen(seed + 3)
        b = _load(case, torch.stack([_grf(gen, n, 2, 1.0, n / 8) for _ in range(2)]).reshape(-1))
        return b, (_Ref(case, c).solve(b) if nu + npr <= 60_000 else None)
    if nu + npr > 60_000 or (case["field"] == "channels" and case["precision"] != "fp64"):
        return None   # dozens of reference V-cycles
    return _Ref(case, c).solve(_vectors(case, seed, n, 1).reshape(-1))
