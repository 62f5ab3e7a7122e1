"""Measured cases of the solver library: the calls its users make, over the sizes they use.

Every case goes through the public Python binding (`paper_0901_3163_gb300.dlz`), one
operation or one whole solve per pass.  The gauge links follow the recipe of `synth/`
(U = exp(0.3 i H), H hermitian traceless Gaussian), made on the GPU.  The solves run at
hopping parameters from 0.20 (the parity tests) to 0.25 (the learned-seed workload), where
a solve takes a few hundred iterations, and to a residual of 1e-11, a tenth of the
library's default, so that two correct programs agree to far better than 1e-9.

The kinds and what they stand for:

  apply     one call of the operator D, D^dag, Q or D^dag D on device vectors: what a user's
            own analysis or Krylov code calls.  FP64, FP32 and bfloat16 storage.
  cg        D-CG on N right-hand sides over a Lan-DR set: the paper's second phase on
            D^dag D, and the headline workload.
  minres    D-MinRes on N right-hand sides over a MinRes-DR set: the second phase on Q.
  eo        the same D-CG through the even-odd operator, with preparation and
            reconstruction.
  multi     D-MinRes on several lattices of uneven size in one call.
  first     the paper's whole method: Lan-DR on the first right-hand side, then D-CG on a
            few more over the set that it made.
  basis     the products of the Krylov basis: the restart V P and the projection V^dag R.
  net       one training pass of the parallel-transport network: forward, backward, the
            weight gradients and the input gradient.
"""
import math

import numpy as np
import torch

from paper_0901_3163_gb300 import dlz

TOL = 1e-11
KAPPA_C = 0.2729          # critical hopping parameter of these links on large lattices
WHICH = {"D": dlz.D, "DDAG": dlz.DDAG, "Q": dlz.Q, "DDAGD": dlz.DDAGD}
DTYPE = {"f64": dlz.F64, "f32": dlz.F32, "bf16": dlz.BF16}


def _case(name, kind, dims, **kw):
    c = dict(name=name, kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], bc_t=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call of the operator: a user's own Krylov loop on a test lattice,
        # where the latency of the call is all that counts
        _case("apply_small", "apply", (8, 8, 8, 8), which="D", dtype="f32", nrhs=1, kappa=0.2),
        # all spin-colour sources of one site through gamma5 D in FP32, on the lattice of
        # the MinRes-DR workload
        _case("apply_batch", "apply", (16, 16, 16, 32), which="Q", dtype="f32", nrhs=12, kappa=0.25),
        # a residual check in FP64 on a lattice of uneven extents, antiperiodic in time
        _case("apply_ragged_f64", "apply", (12, 10, 14, 18), which="DDAGD", dtype="f64", nrhs=3, kappa=0.25, bc_t=-1),
        # D-CG on the sizes of the tests: launches and host work against little arithmetic
        _case("cg_small", "cg", (8, 8, 8, 8), precision="f32", nrhs=4, kappa=0.2, m=40, k=10),
        # the headline workload's second phase: 16 right-hand sides of the 24^3 x 48 lattice
        _case("cg_large", "cg", (24, 24, 24, 48), precision="f32", nrhs=16, kappa=0.24, m=40, k=16),
        # D-CG through the even-odd operator, half a batch
        _case("eo_cg", "eo", (16, 16, 16, 32), precision="f32", nrhs=8, kappa=0.25, m=40, k=16),
        # the 16^3 x 32 workload's second phase: 11 spin-colour point sources at one site
        _case("minres_points", "minres", (16, 16, 16, 32), precision="f32", nrhs=11, kappa=0.25, m=40, k=20,
              source="point"),
        # the plain FP64 form on a lattice of uneven extents
        _case("minres_f64", "minres", (12, 12, 10, 22), precision="f64", nrhs=2, kappa=0.24, m=40, k=10, bc_t=-1),
        # lattices of three sizes in one call, as the uneven multi-lattice workload
        _case("multi_lattice", "multi", (8, 12, 16, 0), nlat=9, nrhs=8, kappa=0.25, m=40, k=10),
        # the whole method, with the Krylov sizes of the 16^3 x 32 workload
        _case("first_rhs", "first", (16, 16, 16, 32), nrhs=4, kappa=0.25, m=100, k=40),
        # the restart and projection of Lan-DR(120, 60), on the 16^3 x 32 lattice
        _case("basis_products", "basis", (16, 16, 16, 32), nin=121, nout=61, nq=16, kappa=0.25),
        # a training pass of the learned-seed network, with its widths and batch
        _case("net_train", "net", (16, 16, 16, 16), nvec=4, w1=12, w2=16, kappa=0.25),
    ]


# ---------------------------------------------------------------- drawn cases
def _extents(rng, vmin, vmax, even):
    """Four extents whose product lies in [vmin, vmax], log-uniform, t the longest on average."""
    for _ in range(1000):
        v = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
        a = v ** 0.25
        e = [max(2, int(round(a * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(4)]
        e[3] = max(2, int(round(e[3] * rng.choice((1.0, 1.0, 1.5, 2.0)))))
        if even:
            e = [max(2, 2 * int(round(x / 2))) for x in e]
        if vmin <= e[0] * e[1] * e[2] * e[3] <= vmax:
            return tuple(e)
    return (8, 8, 8, 8)


def draw(rng):
    kind = rng.choice(("apply", "apply", "cg", "cg", "eo", "minres", "minres", "multi", "first", "basis", "net"))
    bc = rng.choice((1, 1, -1))
    kappa = round(rng.uniform(0.2, 0.25), 4)
    if kind == "apply":
        c = _case("", kind, _extents(rng, 256, 300000, rng.random() < 0.5), which=rng.choice(sorted(WHICH)),
                  dtype=rng.choice(("f32", "f32", "f64", "bf16")), nrhs=rng.choice((1, 1, 2, 3, 5, 8, 12, 16)),
                  kappa=kappa)
    elif kind in ("cg", "minres", "eo"):
        f64 = kind != "eo" and rng.random() < 0.25
        c = _case("", kind, _extents(rng, 256, 20000 if f64 else 250000, kind == "eo" or rng.random() < 0.6),
                  precision="f64" if f64 else "f32", nrhs=rng.randint(1, 3) if f64 else rng.randint(1, 16), kappa=kappa,
                  m=rng.choice((24, 40)), k=rng.choice((4, 10, 16, 20)))
        if kind == "minres":
            c["source"] = rng.choice(("gauss", "point"))
            if c["source"] == "point":
                c["nrhs"] = min(c["nrhs"], 11)
    elif kind == "multi":
        sizes = [rng.choice((4, 5, 6, 8, 9, 10, 12, 14)) for _ in range(3)]
        c = _case("", kind, (sizes[0], sizes[1], sizes[2], 0), nlat=rng.randint(2, 10), nrhs=rng.randint(1, 8),
                  kappa=kappa, m=24, k=rng.choice((4, 10)))
    elif kind == "first":
        m, k = rng.choice(((40, 10), (60, 20), (100, 40), (120, 60)))
        c = _case("", kind, _extents(rng, 2000, 130000, rng.random() < 0.6), nrhs=rng.randint(1, 6), kappa=kappa, m=m, k=k)
    elif kind == "basis":
        k = rng.choice((10, 20, 40, 60, 100))
        c = _case("", kind, _extents(rng, 512, 130000, True), nin=min(128, 2 * k + 1), nout=k + 1,
                  nq=rng.choice((1, 4, 8, 12, 16)), kappa=kappa)
    else:
        c = _case("", kind, _extents(rng, 256, 65536, rng.random() < 0.6), nvec=rng.randint(1, 4),
                  w1=rng.choice((4, 6, 8, 12, 16)), w2=rng.choice((3, 8, 12, 16)), kappa=kappa)
    if kind not in ("multi", "basis", "net"):
        c["bc_t"] = bc
    small = min(_multi_dims(c))[0] ** 4 if kind == "multi" else c["lx"] * c["ly"] * c["lz"] * c["lt"]
    if small < 4000:
        c["kappa"] = min(c["kappa"], 0.22)       # the critical value is lower on small lattices
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _normal(shape, g, dtype=torch.complex128):
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, device="cuda", dtype=real))


def _links(dims, g, eps=0.3):
    """U = exp(i eps H) per link, H hermitian traceless: complex128 [4, V, 3, 3]."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    a = _normal((4 * V, 3, 3), g)
    h = 0.5 * (a + a.mH)
    h = h - (h.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3.0)[:, None, None] * torch.eye(3, device="cuda")
    x = (0.25j * eps) * h                    # exp(4 x) by a Taylor series and two squarings
    u = torch.eye(3, device="cuda", dtype=torch.complex128).expand_as(x)
    for n in range(18, 0, -1):
        u = torch.eye(3, device="cuda", dtype=torch.complex128) + (x @ u) / n
    u = u @ u
    u = u @ u
    return u.reshape(4, V, 3, 3).contiguous()


def _rhs(case, V, g):
    n = case["nrhs"]
    if case.get("source") == "point":
        # spin-colour point sources 1 .. n at the origin (source 0 made the deflation set)
        b = torch.zeros(n, V, 12, dtype=torch.complex128, device="cuda")
        for i in range(n):
            b[i, 0, (i + 1) % 12] = 1.0
        return b.reshape(n, V, 4, 3)
    return _normal((n, V, 4, 3), g)


def _multi_dims(case):
    """The lattices of a multi case: L^4 for L cycling through the three extents."""
    ls = (case["lx"], case["ly"], case["lz"])
    return [(ls[i % 3],) * 4 for i in range(case["nlat"])]


def _net_weights(widths, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(len(widths) - 1):
        shp = (9, widths[i + 1], widths[i], 4, 4)
        w = rng.standard_normal(shp) + 1j * rng.standard_normal(shp)
        out.append((w / math.sqrt(2.0 * 36.0 * widths[i])).astype(np.complex64))
    return out


def _first_set(solver, op, b, case):
    """A deflation set as a user has it from the first right-hand side: two restart cycles."""
    p = dlz.params_default(m=case["m"], k=case["k"], precision=dlz.F32, max_cycles=2, eig_only=1)
    return solver(op, b, p)[1]


def prepare(case, seed):
    kind, kappa = case["kind"], case["kappa"]
    if kind == "multi":
        st = dict(case=case, ops=[], defls=[], Bs=[])
        for i, dims in enumerate(_multi_dims(case)):
            g = _gen(seed, 7 + i)
            V = dims[0] ** 4
            op = dlz.create_operator(dims, _links(dims, g), kappa, 1)
            st["ops"].append(op)
            st["defls"].append(_first_set(dlz.minresdr, op, _normal((V, 4, 3), g), case))
            st["Bs"].append(_rhs(case, V, g))
        st["p"] = dlz.params_default(tol=TOL, precision=dlz.F32)
        return st
    dims, g = _dims(case), _gen(seed)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    st = dict(case=case)
    if kind == "basis":
        L = 12 * V
        scale = 1.0 / math.sqrt(2.0 * L)
        st["V"] = _normal((case["nin"], L), g, torch.complex64) * scale     # near-orthonormal rows
        st["R"] = _normal((case["nq"], L), g, torch.complex64)
        q = np.linalg.qr(np.random.default_rng(seed).standard_normal((case["nin"], case["nout"])))[0]
        st["P"] = np.ascontiguousarray(q)
        return st
    U = _links(dims, g)
    make = dlz.create_operator_eo if kind == "eo" else dlz.create_operator
    op = st["op"] = make(dims, U, kappa, case["bc_t"])
    if kind == "apply":
        ctype = torch.complex128 if case["dtype"] == "f64" else torch.complex64
        st["x"] = _normal((case["nrhs"], V, 4, 3), g, ctype)
        st["out"] = torch.empty_like(st["x"])
    elif kind == "net":
        widths = (1, case["w1"], case["w2"], 1)
        st["net"] = dlz.net_create(op, widths, _net_weights(widths, seed))
        st["x"] = _normal((case["nvec"], V, 4, 3), g, torch.complex64)
        st["g"] = _normal((case["nvec"], V, 4, 3), g, torch.complex64)
    elif kind == "first":
        st["b"] = _normal((V, 4, 3), g)
        st["B"] = _normal((case["nrhs"], V, 4, 3), g)
        st["p"] = dlz.params_default(m=case["m"], k=case["k"], tol=TOL, precision=dlz.F32)
    else:
        n = V // 2 if kind == "eo" else V
        solver = dlz.minresdr if kind == "minres" else dlz.landr
        st["defl"] = _first_set(solver, op, _normal((n, 4, 3), g), case)
        st["B"] = _rhs(case, V, g)
        st["p"] = dlz.params_default(tol=TOL, precision=DTYPE[case["precision"]])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "apply":
        return dlz.apply(st["op"], WHICH[case["which"]], st["x"], st["out"], DTYPE[case["dtype"]])
    if kind == "cg":
        return dlz.dcg(st["op"], st["defl"], st["B"], st["p"])[0]
    if kind == "minres":
        return dlz.dminres(st["op"], st["defl"], st["B"], st["p"])[0]
    if kind == "eo":
        be = dlz.eo_prepare(st["op"], st["B"])
        xe, _ = dlz.dcg(st["op"], st["defl"], be, st["p"])
        return dlz.eo_reconstruct(st["op"], xe, st["B"])
    if kind == "multi":
        return dlz.batch_dminres(st["ops"], st["defls"], st["Bs"], st["p"])[0]
    if kind == "first":
        x, defl, _ = dlz.landr(st["op"], st["b"], st["p"])
        return [x, dlz.dcg(st["op"], defl, st["B"], st["p"])[0]]
    if kind == "basis":
        restart = dlz.basis_combine(torch.view_as_real(st["V"]).reshape(case["nin"], -1), st["P"])
        return [restart, dlz.basis_dots(st["V"], st["R"])]
    net = st["net"]
    dlz.net_zero_grad(net)
    f = dlz.net_forward(net, st["x"])
    gin = dlz.net_backward(net, st["g"], want_input_grad=True)
    return [f, gin] + dlz.net_get(net, 1)


# ---------------------------------------------------------------- work
def _iterations(kappa, residual, per):
    """Steps of CG on the normal equations (per = 1) or MinRes on Q (per = 2) to `residual`."""
    smin = max(1.0 - kappa / KAPPA_C, 0.02)
    cond = (1.0 + kappa / KAPPA_C) / smin
    return 0.5 * per * cond * math.log(2.0 / residual)


def work(case):
    kind = case["kind"]
    if kind == "multi":
        vr = sum(d[0] ** 4 for d in _multi_dims(case)) * case["nrhs"]
        v = vr / case["nrhs"]
        it = _iterations(case["kappa"], TOL, 1.0)
        return {"bytes": v * 576 + vr * 384, "flops": it * vr * (1368 + 12 * 24)}
    V = case["lx"] * case["ly"] * case["lz"] * case["lt"]
    if kind == "apply":
        esz = {"f64": 16, "f32": 8, "bf16": 8}[case["dtype"]]
        link = 576 if case["dtype"] == "f64" else 192
        mv = 2 if case["which"] == "DDAGD" else 1
        return {"bytes": V * (link + 24.0 * esz * case["nrhs"]), "flops": 1368.0 * V * case["nrhs"] * mv}
    if kind == "basis":
        n, o, q = case["nin"], case["nout"], case["nq"]
        return {"bytes": 96.0 * V * (n + o + n + q), "flops": 24.0 * V * (2.0 * n * o + 4.0 * n * q)}
    if kind == "net":
        w = (1, case["w1"], case["w2"], 1)
        mac = sum(9.0 * 48 * a * b for a, b in zip(w, w[1:])) + sum(8.0 * 36 * a for a in w[:-1])
        sv = V * case["nvec"]
        # forward, input gradient and weight gradient; inputs, outputs and the layers'
        # inputs kept for the backward pass
        return {"bytes": V * 192.0 + 96.0 * sv * (4 + 2 * (w[1] + w[2])), "flops": 8.0 * 3 * sv * mac}
    n = case["nrhs"]
    minres = kind == "minres"
    it = _iterations(case["kappa"], TOL, 1.0)
    # per iteration: the stencils (two of D for CG, one for MinRes) and the vector updates
    flops = it * V * n * ((1 if minres else 2) * 1368 + 10 * 24)
    bytes_ = V * (576.0 + 384.0 * n)
    if kind == "eo":
        flops *= 0.5
    if kind == "first":
        flops += V * (it * (2 * 1368 + 10 * 24 + 16 * 24 * case["k"]))
        bytes_ += V * (384.0 + 192.0 * case["k"])
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- 64-bit reference
# Plain torch in complex128: fields [Lt, Lz, Ly, Lx, 3, 4 N] (colour, then right-hand side
# and spin), links as small matrices, gamma matrices as a permutation and a phase.
_GAMMA = (((3, 2, 1, 0), (-1j, -1j, 1j, 1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)),
          ((2, 3, 0, 1), (-1j, 1j, 1j, -1j)), ((2, 3, 0, 1), (1, 1, 1, 1)))


class _Wilson:
    def __init__(self, dims, U, kappa, bc):
        self.shape = (dims[3], dims[2], dims[1], dims[0])
        self.U = [U[mu].reshape(self.shape + (3, 3)) for mu in range(4)]
        self.kappa = kappa
        if bc == -1:
            self.U[3] = self.U[3].clone()
            self.U[3][-1] *= -1.0
        self.g = [(torch.tensor(p, device="cuda"), torch.tensor(f, device="cuda", dtype=torch.complex128))
                  for p, f in _GAMMA]

    def gam(self, mu, v):
        p, f = self.g[mu]
        w = v.reshape(self.shape + (3, -1, 4))
        return (w[..., p] * f).reshape(v.shape)

    def g5(self, v):
        s = torch.tensor([1.0, 1.0, -1.0, -1.0], device="cuda")
        return (v.reshape(self.shape + (3, -1, 4)) * s).reshape(v.shape)

    def hop(self, v):
        acc = torch.zeros_like(v)
        for mu in range(4):
            ax = 3 - mu
            f = self.U[mu] @ torch.roll(v, -1, ax)
            acc += f - self.gam(mu, f)
            b = torch.roll(self.U[mu].mH @ v, 1, ax)
            acc += b + self.gam(mu, b)
        return acc

    def D(self, v):
        return v - self.kappa * self.hop(v)

    def Ddag(self, v):
        return self.g5(self.D(self.g5(v)))

    def into(self, b):
        """[N, V, 4, 3] -> fields"""
        n = b.shape[0]
        return b.reshape((n,) + self.shape + (4, 3)).permute(1, 2, 3, 4, 6, 0, 5).reshape(self.shape + (3, 4 * n)).contiguous()

    def outof(self, v):
        n = v.shape[-1] // 4
        return v.reshape(self.shape + (3, n, 4)).permute(5, 0, 1, 2, 3, 6, 4).reshape(n, -1, 4, 3).contiguous()

    def dots(self, a, b):
        n = a.shape[-1] // 4
        return (a.conj() * b).real.reshape(-1, n, 4).sum((0, 2))

    def solve(self, b):
        """D x = b by conjugate gradients on the normal equations, restarted from the true residual."""
        x = torch.zeros_like(b)
        wide = lambda c: c.repeat_interleave(4)      # noqa: E731  one factor per right-hand side
        bb = self.dots(b, b).clamp_min(1e-300)
        for _ in range(4):
            s = b - self.D(x)
            if bool((self.dots(s, s) <= 1e-28 * bb).all()):
                break
            r = self.Ddag(s)
            p, rr = r.clone(), self.dots(r, r)
            r0 = rr.clone().clamp_min(1e-300)
            for it in range(1500):
                t = self.D(p)
                al = rr / self.dots(t, t).clamp_min(1e-300)
                x += wide(al) * p
                r -= wide(al) * self.Ddag(t)
                rn = self.dots(r, r)
                p = r + wide(rn / rr.clamp_min(1e-300)) * p
                rr = rn
                if it % 16 == 15 and bool((rr <= 1e-28 * r0).all()):
                    break
        return x


def _exact_net(W, U, dims, x, gout):
    """Forward and gradients G(z) = dL/dRe z + i dL/dIm z of the network, weights rounded to bfloat16."""
    shape = (dims[3], dims[2], dims[1], dims[0])
    us = [U[mu].reshape(shape + (3, 3)) for mu in range(4)]
    Wb = []
    for w in W:
        t = torch.view_as_real(torch.from_numpy(w)).to(torch.bfloat16).to(torch.float64)
        Wb.append(torch.view_as_complex(t.contiguous()).cuda())

    def move(v, o, adj=False):                   # v [C, T, Z, Y, X, 3, 4]
        if o == 0:
            return v
        mu, fwd = (o - 1) // 2, (o - 1) % 2 == 0
        ax = 1 + 3 - mu
        if fwd != adj:
            return us[mu] @ torch.roll(v, -1, ax)
        return torch.roll(us[mu].mH @ v, 1, ax)

    fs, gins = [], []
    grads = [torch.zeros_like(w) for w in Wb]
    for i in range(x.shape[0]):
        to = lambda t: t.to(torch.complex128).reshape((1,) + shape + (4, 3)).transpose(-1, -2).contiguous()  # noqa: E731
        acts = [to(x[i])]
        for w in Wb:
            out = 0
            for o in range(9):
                out = out + torch.einsum("dcst,c...t->d...s", w[o], move(acts[-1], o))
            acts.append(out)
        g = to(gout[i])
        for li in range(len(Wb) - 1, -1, -1):
            w, a = Wb[li], acts[li]
            gi = 0
            for o in range(9):
                t = move(a, o)
                grads[li][o] += torch.einsum("das,cat->dcst", g.reshape(g.shape[0], -1, 4), t.reshape(t.shape[0], -1, 4).conj())
                gi = gi + move(torch.einsum("dcst,d...s->c...t", w[o].conj(), g), o, adj=True)
            g = gi
        back = lambda t: t.transpose(-1, -2).reshape(-1, 4, 3)  # noqa: E731
        fs.append(back(acts[-1][0]))
        gins.append(back(g[0]))
    return [torch.stack(fs), torch.stack(gins)] + [t.cpu().numpy() for t in grads]


def exact(case, seed):
    kind = case["kind"]
    if kind == "multi":
        out = []
        for i, dims in enumerate(_multi_dims(case)):
            g = _gen(seed, 7 + i)
            w = _Wilson(dims, _links(dims, g), case["kappa"], 1)
            _normal((dims[0] ** 4, 4, 3), g)
            out.append(w.outof(w.solve(w.into(_rhs(case, dims[0] ** 4, g)))))
        return out
    dims, g = _dims(case), _gen(seed)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    if kind == "basis":
        L = 12 * V
        v = _normal((case["nin"], L), g, torch.complex64) * (1.0 / math.sqrt(2.0 * L))
        r = _normal((case["nq"], L), g, torch.complex64)
        q = np.linalg.qr(np.random.default_rng(seed).standard_normal((case["nin"], case["nout"])))[0]
        P = torch.from_numpy(q).cuda()
        vr = torch.view_as_real(v).reshape(case["nin"], -1)
        restart = torch.cat([P.T @ c.double() for c in vr.split(1 << 20, dim=1)], dim=1)
        dots = sum(b.to(torch.complex128) @ a.to(torch.complex128).mH
                   for a, b in zip(v.split(1 << 19, dim=1), r.split(1 << 19, dim=1)))
        return [restart, dots]
    U = _links(dims, g)
    if kind == "net":
        W = _net_weights((1, case["w1"], case["w2"], 1), seed)
        x = _normal((case["nvec"], V, 4, 3), g, torch.complex64)
        gout = _normal((case["nvec"], V, 4, 3), g, torch.complex64)
        return _exact_net(W, U, dims, x, gout)
    w = _Wilson(dims, U, case["kappa"], case["bc_t"])
    if kind == "apply":
        x = _normal((case["nrhs"], V, 4, 3), g, torch.complex128 if case["dtype"] == "f64" else torch.complex64)
        if case["dtype"] == "bf16":
            x = torch.view_as_complex(torch.view_as_real(x).to(torch.bfloat16).float())
        v = w.into(x.to(torch.complex128))
        out = {"D": w.D, "DDAG": w.Ddag, "Q": lambda t: w.g5(w.D(t)),
               "DDAGD": lambda t: w.Ddag(w.D(t))}[case["which"]](v)
        return w.outof(out)
    if V * case["nrhs"] > 4000000:
        return None                              # more than about 20 seconds
    if kind == "first":
        b = _normal((V, 4, 3), g)
        B = _normal((case["nrhs"], V, 4, 3), g)
        x = w.outof(w.solve(w.into(torch.cat([b[None], B]))))
        return [x[0], x[1:].contiguous()]
    _normal((V // 2 if kind == "eo" else V, 4, 3), g)
    return w.outof(w.solve(w.into(_rhs(case, V, g))))
