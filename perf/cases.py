"""What a user of this library has it compute, as timed and compared workloads.

Families (the "do" of a case):

* ``local``    one ``ax_local``: the element operator Y_e = D^T (w G) D X_e (Algorithm 1), the call every solver
               iteration and every benchmark makes.  Orders, geometry kinds and precisions of the order sweep.
* ``pcg``      a whole ``pcg_solve`` of an assembled Dirichlet Poisson problem to 1e-10 (Eq. 1).
* ``mixed``    the same solve by ``pcg_solve_mixed``: FP64 refinement around a float32 inner solver.
* ``batch``    ``ax_batch_pcg`` on many meshes of uneven size and order, a fixed number of iterations.
* ``forward``  the learned preconditioner's network on a row per element (``ax_mlp_forward``).
* ``grad``     its loss and gradients on a mini-batch (``ax_mlp_grad``), the step training repeats.

Meshes are the perturbed boxes and the boxes of parallelepipeds of the benchmark, every one drawn from the seed.
``exact`` is plain torch in float64: the Gauss-Lobatto-Legendre rule, the trilinear Jacobian and the operator are
written out again below.
"""
import math

import numpy as np
import torch

from paper_2504_07042_gb300 import ax, inputs

DEV = "cuda:0"
F64IO = ("fp64", "f64dw")
IN, IN_PAD, HID, OUT = 536, 544, 512, 512  # the network's sizes (AxMLP)
TOL = 1e-10                                # solves: the tolerance the solvers are compared with the oracle at


# ------------------------------------------------------------------------------------------------ the cases

def listed():
    return [
        # the headline of the order sweep: FP64-accurate recompute on 67.1M local nodes
        _local("local_f64dw_trilinear_n7", "f64dw", "trilinear", 7, 64, 64, 32),
        # the parity mesh, 512 elements: one call of a small problem, where latency and launches count
        _local("local_f64dw_trilinear_n7_small", "f64dw", "trilinear", 7, 8, 8, 8),
        # a higher order with affine elements (structured meshes), a ragged count of elements per SM
        _local("local_f64dw_parallelepiped_n11", "f64dw", "parallelepiped", 11, 34, 34, 34),
        # single precision at the default order: smoothers, inner solvers
        _local("local_fp32_trilinear_n7", "fp32", "trilinear", 7, 64, 64, 32),
        # the stored-factor baseline in single precision, order 5, odd sizes
        _local("local_fp32_stored_n5", "fp32", "stored", 5, 68, 68, 67),
        # tensor-core contractions at the highest order of the sweep
        _local("local_bf16_trilinear_n15", "bf16", "trilinear", 15, 32, 32, 16),
        # the binding's default precision on a mid-size mesh with odd dimensions
        _local("local_fp64_trilinear_n4_odd", "fp64", "trilinear", 4, 33, 21, 17),
        # the FP64-accurate Jacobi-PCG on 16^3 elements of order 7
        {"name": "pcg_f64dw_n7", "do": "pcg", "prec": "f64dw", "N": 7, "ex": 16, "ey": 16, "ez": 16},
        # the fastest solver of the same problem
        {"name": "mixed_f64dw_fp32_n7", "do": "mixed", "prec": "f64dw", "lo": "fp32", "N": 7, "ex": 16, "ey": 16,
         "ez": 16},
        # sixteen meshes of orders 3 to 9 advanced together
        {"name": "batch_fp32_16", "do": "batch", "meshes": 16, "seed_e": 4, "seed_n": 5, "iters": 20},
        # the network on every element of the 32^3 mesh of the learned solver
        {"name": "mlp_forward_32768", "do": "forward", "rows": 32768},
        # one mini-batch of its training
        {"name": "mlp_grad_4096", "do": "grad", "rows": 4096},
    ]


def _local(name, prec, kind, N, ex, ey, ez):
    return {"name": name, "do": "local", "prec": prec, "kind": kind, "N": N, "ex": ex, "ey": ey, "ez": ez}


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, elements):
    """Three box dimensions of about that many elements, odd and even ones."""
    a = max(1.0, elements ** (1.0 / 3.0))
    ex = max(1, round(a * rng.uniform(0.8, 1.25)))
    ey = max(1, round(a * rng.uniform(0.8, 1.25)))
    return ex, ey, max(1, round(elements / (ex * ey)))


def draw(rng):
    do = rng.choice(["local"] * 7 + ["pcg", "mixed", "batch", "forward", "grad"])
    if do == "local":
        prec = rng.choice(["f64dw", "f64dw", "f64dw", "fp32", "fp32", "tf32", "bf16", "fp16", "fp64"])
        kind = rng.choice(["trilinear", "trilinear", "parallelepiped", "stored", "partial"])
        N = rng.randint(3, 15)
        nodes = _log(rng, 2.5e5, 6.0e6 if prec == "fp64" else 6.4e7)
        ex, ey, ez = _box(rng, nodes / (N + 1) ** 3)
        c = _local("", prec, kind, N, ex, ey, ez)
        del c["name"]
        return c
    if do in ("pcg", "mixed"):
        N = rng.randint(3, 9)
        ex, ey, ez = _box(rng, _log(rng, 5.0e4, 1.3e6) / N ** 3)
        c = {"do": do, "prec": "f64dw", "N": N, "ex": ex, "ey": ey, "ez": ez}
        if do == "mixed":
            c["lo"] = rng.choice(["fp32", "fp32", "tf32", "bf16", "fp16"])
        return c
    if do == "batch":
        return {"do": "batch", "meshes": rng.randint(4, 16), "seed_e": rng.randint(6, 999),
                "seed_n": rng.randint(6, 999), "iters": rng.randint(8, 20)}
    if do == "forward":
        return {"do": "forward", "rows": round(_log(rng, 100, 32768))}
    return {"do": "grad", "rows": 32 * round(_log(rng, 8, 256))}


# ------------------------------------------------------------------------------------- what a program has in hand

def _vertices(c, seed):
    if c.get("kind") == "parallelepiped":
        return inputs.parallelepiped_vertices(c["ex"], c["ey"], c["ez"], 2 + 2 * seed, 3 + 2 * seed)
    return inputs.box_vertices(c["ex"], c["ey"], c["ez"], 0.1, seed)


def _io(prec):
    return torch.float64 if prec in F64IO else torch.float32


def _rand(shape, seed, lo=-1.0, hi=1.0, dtype=torch.float64):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * (seed % 1000003) + 17)
    return torch.rand(shape, generator=g, device=DEV, dtype=dtype) * (hi - lo) + lo


def _source(xyz, seed):
    """A smooth source on the box: a short random sine series (xyz [E][3][n3])."""
    k = np.random.default_rng(seed).standard_normal((3, 3, 3))
    f = torch.zeros_like(xyz[:, 0])
    top = xyz.amax(dim=(0, 2))
    s = [[torch.sin((a + 1) * math.pi * xyz[:, d] / top[d]) for a in range(3)] for d in range(3)]
    for a in range(3):
        for b in range(3):
            for e in range(3):
                f += float(k[a, b, e]) / ((a + 1) ** 2 + (b + 1) ** 2 + (e + 1) ** 2) * s[0][a] * s[1][b] * s[2][e]
    return f


def _numbering(ex, ey, ez, N):
    """Global ids [E][(N+1)^3] and the boundary mask of a box (x fastest), on the GPU."""
    ar = lambda n: torch.arange(n, device=DEV)  # noqa: E731
    gx, gy, gz = ex * N + 1, ey * N + 1, ez * N + 1
    X = (ar(ex) * N)[:, None] + ar(N + 1)[None, :]
    Y = (ar(ey) * N)[:, None] + ar(N + 1)[None, :]
    Z = (ar(ez) * N)[:, None] + ar(N + 1)[None, :]
    gid = (Z[:, None, None, :, None, None] * (gx * gy) + Y[None, :, None, None, :, None] * gx
           + X[None, None, :, None, None, :]).reshape(ex * ey * ez, (N + 1) ** 3).contiguous()
    m = torch.zeros((gz, gy, gx), dtype=torch.uint8, device=DEV)
    m[0], m[-1] = 1, 1
    m[:, 0], m[:, -1] = 1, 1
    m[:, :, 0], m[:, :, -1] = 1, 1
    return gid, gx * gy * gz, m.reshape(-1)


def _mesh_list(c, seed):
    out = []
    for q, (ex, ey, ez, N) in enumerate(inputs.batch_meshes(c["meshes"], c["seed_e"], c["seed_n"])):
        V = torch.from_numpy(inputs.box_vertices(ex, ey, ez, 0.1, 100 * seed + q)).to(DEV)
        out.append((V, N) + _numbering(ex, ey, ez, N))
    return out


def _weights(seed):
    """Network parameters of the size training starts from, small random biases."""
    g = torch.Generator(device=DEV)
    g.manual_seed(7919 * (seed % 1000003) + 3)
    n = lambda *s: torch.randn(s, generator=g, device=DEV)  # noqa: E731
    W1 = n(HID, IN_PAD) * math.sqrt(2.0 / IN)
    W1[:, IN:] = 0.0
    parts = [W1, 0.1 * n(HID), n(HID, HID) * math.sqrt(2.0 / HID), 0.1 * n(HID), n(OUT, HID) / math.sqrt(HID),
             0.1 * n(OUT)]
    return parts


def _features(rows, seed):
    X = _rand((rows, IN_PAD), seed, dtype=torch.float32)
    X[:, IN:] = 0.0
    return X.to(torch.bfloat16)


def prepare(case, seed):
    c, do = case, case["do"]
    if do == "local":
        op = ax.Ax(torch.from_numpy(_vertices(c, seed)).to(DEV), c["N"], c["kind"], c["prec"])
        X = _rand((op.E, op.n3), seed, dtype=_io(c["prec"]))
        return {"do": do, "op": op, "X": X, "Y": torch.empty_like(X)}
    if do in ("pcg", "mixed"):
        V = torch.from_numpy(_vertices(c, seed)).to(DEV)
        op = ax.Ax(V, c["N"], "trilinear", c["prec"])
        gid, ng, mask = _numbering(c["ex"], c["ey"], c["ez"], c["N"])
        op.gs_setup(gid, ng, mask)
        xyz = op.ax_node_coords(torch.empty((op.E, 3, op.n3), dtype=torch.float64, device=DEV))
        f = _source(xyz, seed)
        b = op.gs_gather(op.ax_mass(f, torch.empty_like(f)), torch.empty(ng, dtype=torch.float64, device=DEV))
        s = {"do": do, "op": op, "b": b, "x": torch.empty_like(b)}
        if do == "mixed":
            s["lo"] = ax.Ax(V, c["N"], "trilinear", c["lo"])
            s["inner"] = 1e-3 if c["lo"] == "fp32" else 1e-2
        return s
    if do == "batch":
        bt = ax.AxBatch(_mesh_list(c, seed), "trilinear", "fp32")
        b = _rand((bt.n_global,), seed, 0.5, 1.5, torch.float32)
        return {"do": do, "bt": bt, "b": b, "x": torch.empty_like(b), "iters": c["iters"]}
    mlp = ax.AxMLP(seed=0)
    mlp.ax_mlp_set_params(torch.cat([p.reshape(-1) for p in _weights(seed)]))
    s = {"do": do, "mlp": mlp, "X": _features(c["rows"], seed)}
    if do == "forward":
        s["Y"] = torch.empty((c["rows"], OUT), dtype=torch.float32, device=DEV)
    else:
        s["T"] = _rand((c["rows"], OUT), seed + 1, dtype=torch.float32)
        s["g"] = torch.empty(mlp.num_params, dtype=torch.float32, device=DEV)
    return s


def run(state):
    s, do = state, state["do"]
    if do == "local":
        return s["op"].ax_local(s["X"], s["Y"])
    if do == "pcg":
        s["op"].pcg_solve(s["b"], s["x"].zero_(), rtol=TOL, maxit=20000, precond=1)
        return s["x"]
    if do == "mixed":
        s["op"].pcg_solve_mixed(s["lo"], s["b"], s["x"].zero_(), rtol=TOL, inner_rtol=s["inner"], max_outer=100)
        return s["x"]
    if do == "batch":
        s["bt"].ax_batch_pcg(s["b"], s["x"].zero_(), rtol=0.0, maxit=s["iters"], graph=1)
        return s["x"]
    if do == "forward":
        return s["mlp"].ax_mlp_forward(s["X"], s["Y"])
    loss, g = s["mlp"].ax_mlp_grad(s["X"], s["T"], s["g"])
    return {"loss": loss, "grads": g}


# -------------------------------------------------------------------------------------------- unavoidable work

def _local_work(E, N, kind, word):
    n3 = (N + 1) ** 3
    geo = {"stored": 6 * n3, "trilinear": 24, "parallelepiped": 8, "partial": n3 + 24}[kind]
    return E * (2 * n3 + geo) * word, E * (12.0 * (N + 1) ** 4 + 15.0 * n3)


def _cg_work(E, N, ng, word, iters):
    """CG iterations: the element operator, five vectors read and four written, the numbering read twice."""
    by, fl = _local_work(E, N, "trilinear", word)
    return iters * (by + 9 * ng * word + 8.0 * E * (N + 1) ** 3), iters * (fl + 14.0 * ng)


def work(case):
    c, do = case, case["do"]
    if do == "local":
        by, fl = _local_work(c["ex"] * c["ey"] * c["ez"], c["N"], c["kind"], 8 if c["prec"] in F64IO else 4)
    elif do in ("pcg", "mixed"):
        # Jacobi-PCG to 1e-10 takes about 6 max(ex, ey, ez) N iterations on these boxes
        e = (c["ex"], c["ey"], c["ez"])
        ng = math.prod(v * c["N"] + 1 for v in e)
        by, fl = _cg_work(math.prod(e), c["N"], ng, 8 if do == "pcg" else 4, 6.0 * max(e) * c["N"])
    elif do == "batch":
        by = fl = 0.0
        for ex, ey, ez, N in inputs.batch_meshes(c["meshes"], c["seed_e"], c["seed_n"]):
            ng = (ex * N + 1) * (ey * N + 1) * (ez * N + 1)
            b, f = _cg_work(ex * ey * ez, N, ng, 4, c["iters"])
            by, fl = by + b, fl + f
    else:
        M, nw = c["rows"], IN_PAD * HID + HID * HID + HID * OUT
        by, fl = M * (2.0 * IN_PAD + 4 * OUT) + 2.0 * nw, 2.0 * M * nw
        if do == "grad":
            by, fl = by + 4.0 * nw, fl + 2.0 * M * nw + 2.0 * M * (HID * HID + HID * OUT)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------------------------ in 64 bits

def _gll(N):
    """Points, weights and the differentiation matrix of the Gauss-Lobatto-Legendre rule."""
    c = np.zeros(N + 1)
    c[N] = 1.0
    L = np.polynomial.legendre
    x = np.concatenate([[-1.0], np.sort(np.real(L.legroots(L.legder(c)))) if N > 1 else [], [1.0]])
    for _ in range(3):  # Newton on the interior points
        p1, p2 = L.legval(x[1:-1], L.legder(c)), L.legval(x[1:-1], L.legder(c, 2))
        x[1:-1] -= p1 / p2
    x = 0.5 * (x - x[::-1])
    P = L.legval(x, c)
    w = 2.0 / (N * (N + 1) * P ** 2)
    D = np.zeros((N + 1, N + 1))
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = P[i] / (P[j] * (x[i] - x[j]))
    D[0, 0], D[N, N] = -N * (N + 1) / 4.0, N * (N + 1) / 4.0
    t = lambda a: torch.from_numpy(a).to(DEV)  # noqa: E731
    return t(x), t(w), t(D)


class _Reference:
    """The element operator of one mesh, node (i, j, k) of an element at [k][j][i]."""

    def __init__(self, V, N):
        self.V = V if isinstance(V, torch.Tensor) else torch.from_numpy(V).to(DEV)
        self.N, self.E = N, self.V.shape[0]
        self.x, self.w, self.D = _gll(N)
        self.step = max(1, (1 << 22) // (N + 1) ** 3)
        lo, hi = 0.5 * (1 - self.x), 0.5 * (1 + self.x)
        self.l = torch.stack([lo, hi])           # the two linear shape functions at the points
        self.dl = torch.tensor([-0.5, 0.5], dtype=torch.float64, device=DEV)

    def _corners(self, V):
        return V.reshape(-1, 2, 2, 2, 3)          # [e][c][b][a][coordinate]

    def coords(self):
        X = torch.einsum("ecbax,ck,bj,ai->exkji", self._corners(self.V), self.l, self.l, self.l)
        return X.reshape(self.E, 3, -1)

    def factors(self, V):
        """The six factors of G = w |J| J^-1 J^-T and w |J|, each [e][k][j][i]."""
        C, l, n = self._corners(V), self.l, self.N + 1
        Jr = torch.einsum("ecbax,ck,bj,a->ekjx", C, l, l, self.dl)[:, :, :, None].expand(-1, n, n, n, 3)
        Js = torch.einsum("ecbax,ck,b,ai->ekix", C, l, self.dl, l)[:, :, None].expand(-1, n, n, n, 3)
        Jt = torch.einsum("ecbax,c,bj,ai->ejix", C, self.dl, l, l)[:, None].expand(-1, n, n, n, 3)
        a, b, c = torch.linalg.cross(Js, Jt), torch.linalg.cross(Jt, Jr), torch.linalg.cross(Jr, Js)
        det = (Jr * a).sum(-1)
        w3 = self.w[:, None, None] * self.w[None, :, None] * self.w[None, None, :]
        s = w3 / det
        g = [(p * q).sum(-1) * s for p, q in ((a, a), (a, b), (a, c), (b, b), (b, c), (c, c))]
        return g, w3 * det

    def local(self, X):
        n, D, out = self.N + 1, self.D, torch.empty((self.E, (self.N + 1) ** 3), dtype=torch.float64, device=DEV)
        for e in range(0, self.E, self.step):
            u = X[e:e + self.step].double().reshape(-1, n, n, n)
            g, _ = self.factors(self.V[e:e + self.step])
            ur, us, ut = u @ D.T, D @ u, torch.einsum("kn,enji->ekji", D, u)
            r = g[0] * ur + g[1] * us + g[2] * ut
            s = g[1] * ur + g[3] * us + g[4] * ut
            t = g[2] * ur + g[4] * us + g[5] * ut
            y = r @ D + D.T @ s + torch.einsum("nk,enji->ekji", D, t)
            out[e:e + self.step] = y.reshape(-1, n ** 3)
        return out

    def mass(self, F):
        out = torch.empty_like(F)
        for e in range(0, self.E, self.step):
            out[e:e + self.step] = self.factors(self.V[e:e + self.step])[1].reshape(F[e:e + self.step].shape) * F[e:e + self.step]
        return out

    def diagonal(self):
        n, D, out = self.N + 1, self.D, torch.empty((self.E, (self.N + 1) ** 3), dtype=torch.float64, device=DEV)
        D2, d = D * D, torch.diagonal(D)
        for e in range(0, self.E, self.step):
            g, _ = self.factors(self.V[e:e + self.step])
            y = g[0] @ D2 + D2.T @ g[3] + torch.einsum("nk,enji->ekji", D2, g[5])
            y += 2 * (g[1] * d[None, :, None] * d + g[2] * d[:, None, None] * d + g[4] * d[:, None, None] * d[:, None])
            out[e:e + self.step] = y.reshape(-1, n ** 3)
        return out


def _gather(gid, ng, Y, mask):
    y = torch.zeros(ng, dtype=torch.float64, device=DEV).index_add_(0, gid.reshape(-1), Y.reshape(-1))
    y[mask.bool()] = 0.0
    return y


def _cg(ref, gid, ng, mask, b, rtol, maxit):
    """Jacobi-preconditioned conjugate gradients from zero."""
    A = lambda v: _gather(gid, ng, ref.local(v[gid]), mask)  # noqa: E731
    dg = _gather(gid, ng, ref.diagonal(), mask)
    inv = torch.where(mask.bool(), torch.zeros_like(dg), 1.0 / dg)
    x, r = torch.zeros_like(b), torch.where(mask.bool(), torch.zeros_like(b), b)
    z = inv * r
    p, rz, stop = z.clone(), torch.dot(r, z), rtol * float(r.norm())
    for _ in range(maxit):
        w = A(p)
        alpha = rz / torch.dot(p, w)
        x += alpha * p
        r -= alpha * w
        if rtol and float(r.norm()) <= stop:
            break
        z = inv * r
        new = torch.dot(r, z)
        p = z + (new / rz) * p
        rz = new
    return x


def _network(rows, seed):
    """The parameters as the tensor cores see them (weights in bfloat16), and the features, in 64 bits."""
    P = _weights(seed)
    P = [(p.to(torch.bfloat16) if p.dim() == 2 else p).double() for p in P]
    return P, _features(rows, seed).double()


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z * math.sqrt(0.5)))


def _gelu_grad(z):
    return 0.5 * (1.0 + torch.erf(z * math.sqrt(0.5))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi)


def exact(case, seed):
    c, do = case, case["do"]
    if do == "local":
        ref = _Reference(_vertices(c, seed), c["N"])
        return ref.local(_rand((ref.E, (c["N"] + 1) ** 3), seed, dtype=_io(c["prec"])))
    if do in ("pcg", "mixed"):
        ref = _Reference(_vertices(c, seed), c["N"])
        gid, ng, mask = _numbering(c["ex"], c["ey"], c["ez"], c["N"])
        b = _gather(gid, ng, ref.mass(_source(ref.coords(), seed)), mask)
        return _cg(ref, gid, ng, mask, b, 1e-13, 4000)
    if do == "batch":
        meshes = _mesh_list(c, seed)
        b = _rand((sum(m[3] for m in meshes),), seed, 0.5, 1.5, torch.float32).double()
        out, at = [], 0
        for V, N, gid, ng, mask in meshes:
            out.append(_cg(_Reference(V, N), gid, ng, mask, b[at:at + ng], 0.0, c["iters"]))
            at += ng
        return torch.cat(out)
    (W1, b1, W2, b2, W3, b3), X = _network(c["rows"], seed)
    z1 = X @ W1.T + b1
    h1 = _gelu(z1)
    z2 = h1 @ W2.T + b2
    h2 = _gelu(z2)
    Y = h2 @ W3.T + b3
    if do == "forward":
        return Y
    d3 = (Y - _rand((c["rows"], OUT), seed + 1, dtype=torch.float32).double()) / Y.numel()
    loss = 0.5 * float(d3.square().sum()) * Y.numel()
    d2 = (d3 @ W3) * _gelu_grad(z2)
    d1 = (d2 @ W2) * _gelu_grad(z1)
    grads = [d1.T @ X, d1.sum(0), d2.T @ h1, d2.sum(0), d3.T @ h2, d3.sum(0)]
    return {"loss": loss, "grads": torch.cat([g.reshape(-1) for g in grads])}
