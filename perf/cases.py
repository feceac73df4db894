"""The work a user of this solver library has it do, as timed cases.

Every case goes through the public entry points of the Python binding on fields that live on
the GPU.  The kinds of work, from the inside of a solve to the whole of it:

  apply  one application of the Wilson-clover operator A (residual checks, a user's own
         Krylov loop, several right-hand sides at once)
  sap    one application of the Schwarz preconditioner M (a user's own outer solver)
  setup  a new gauge configuration: load the links, build the clover term, and the first
         FP64 residual and preconditioner application on it
  solve  A x = f to 1e-10 with the deflated FGMRES around M, one or several sources

Lattices, couplings, domain shapes and solver parameters are those of the package's
workloads (8^4, 16^3x32, 24^3x48, 32^3x64) and, in draw(), any allowed lattice between the
smallest and the largest of them.  Gauge fields are random SU(3) links smoothed by APE
smearing (rough ones on 8^4), sources are Gaussian.  exact() restates everything in plain
torch in FP64.
"""
import math

import torch

from paper_1412_2629_gb300 import dd

PREC = {"fp64": dd.DD_PREC_FP64, "fp32": dd.DD_PREC_FP32, "fp16": dd.DD_PREC_FP16, "fp16_h2": dd.DD_PREC_FP16_H2}
REAL_BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "fp16_h2": 2}

# APE smoothed fields are almost free: their critical kappa is 0.125, and 0.124 is the coupling
# of the package's larger workloads; the rough 8^4 field takes 0.130
SMOOTH = {"width": 0.5, "smear": 5, "kappa": 0.124, "csw": 1.5}
ROUGH = {"width": 0.6, "smear": 0, "kappa": 0.130, "csw": 1.0}


def lattice(lx, ly, lz, lt, domain, field):
    bx, by, bz, bt = domain
    return dict(lx=lx, ly=ly, lz=lz, lt=lt, bx=bx, by=by, bz=bz, bt=bt, **field)


def listed():
    c8 = lattice(8, 8, 8, 8, (4, 4, 4, 4), ROUGH)
    c16 = lattice(16, 16, 16, 32, (4, 4, 8, 4), SMOOTH)
    c24 = lattice(24, 24, 24, 48, (4, 4, 4, 4), SMOOTH)
    c32 = lattice(32, 32, 32, 64, (8, 4, 4, 4), SMOOTH)
    return [
        # the smallest operator call, in the layout a user's fields have: latency and launches
        dict(c8, name="apply_fp32_8", kind="apply", prec="fp32", layout="canonical", nrhs=1),
        # the outer solver's operator on the benchmark lattice, fields kept in the library's layout
        dict(c32, name="apply_fp32_32x64", kind="apply", prec="fp32", layout="internal", nrhs=1),
        # the FP64 operator with which a user checks a residual, on the user's own fields
        dict(c24, name="apply_fp64_24x48", kind="apply", prec="fp64", layout="canonical", nrhs=1),
        # the operator on the sources of a batched analysis
        dict(c24, name="apply_fp32_batch_24x48", kind="apply", prec="fp32", layout="internal", nrhs=6),
        # the paper's Schwarz settings on the smallest lattice: 32 short half-sweeps
        dict(c8, name="sap_fp16_8", kind="sap", prec="fp16", layout="internal", nrhs=1, i_s=16, i_d=4, additive=False),
        # single-precision preconditioner on the user's own fields, the domain shape and
        # settings that the autotuner finds for this lattice
        dict(c16, name="sap_fp32_16x32", kind="sap", prec="fp32", layout="canonical", nrhs=1, i_s=4, i_d=4, additive=False),
        # the benchmark's preconditioner: half storage, the largest lattice
        dict(c32, name="sap_fp16_32x64", kind="sap", prec="fp16", layout="internal", nrhs=1, i_s=2, i_d=4, additive=False),
        # several sources per launch, an odd number of them
        dict(c24, name="sap_fp16_batch_24x48", kind="sap", prec="fp16", layout="internal", nrhs=5, i_s=4, i_d=3, additive=False),
        # a new gauge configuration of an ensemble
        dict(c24, name="setup_24x48", kind="setup"),
        # the smallest solve: four steps, bound by latency
        dict(c8, name="solve_8", kind="solve", prec="fp16", nrhs=1, i_s=16, i_d=4, m=16, k=0, steps=4),
        # sources of a batched analysis solved in lockstep with the autotuned settings
        dict(c24, name="solve_batch_24x48", kind="solve", prec="fp16", nrhs=4, i_s=4, i_d=3, m=16, k=6, steps=24),
        # one solve on the benchmark lattice with the benchmark's solver
        dict(c32, name="solve_32x64", kind="solve", prec="fp16", nrhs=1, i_s=2, i_d=4, m=40, k=8, steps=58),
    ]


SHAPES = [(4, 4, 4, 4), (8, 4, 4, 4), (4, 4, 4, 8), (4, 4, 8, 4), (4, 8, 4, 4), (8, 4, 4, 2), (4, 4, 4, 2), (2, 4, 4, 4),
          (8, 8, 2, 4), (2, 4, 8, 8), (4, 4, 2, 2), (16, 4, 2, 4)]


def draw_lattice(rng, largest):
    """An allowed lattice whose volume is spread over the logarithm between 8^4 and `largest`
    sites, its extents multiples (often odd ones) of twice the domain's."""
    want = 4096 * (largest / 4096) ** rng.random()
    for _ in range(1000):
        b = SHAPES[rng.randrange(len(SHAPES))]
        ext = [2 * e * rng.randint(1, 6) for e in b]
        if max(ext) <= 64 and 0.6 * want <= math.prod(ext) <= min(1.5 * want, largest):
            return lattice(*ext, b, SMOOTH)
    return lattice(16, 16, 16, 32, (4, 4, 4, 4), SMOOTH)


def draw(rng):
    kind = rng.choice(["apply", "apply", "sap", "sap", "sap", "setup", "solve"])
    if kind == "apply":
        c = draw_lattice(rng, 32 ** 3 * 64)
        prec = rng.choice(["fp64", "fp32", "fp32", "fp16"])
        layout = "internal" if prec == "fp16" else rng.choice(["internal", "canonical"])
        nrhs = rng.choice([1, 1, 2, 3, 7]) if layout == "internal" and prec != "fp64" and volume(c) <= 700000 else 1
        return dict(c, kind=kind, prec=prec, layout=layout, nrhs=nrhs)
    if kind == "sap":
        c = draw_lattice(rng, 32 ** 3 * 64)
        prec = rng.choice(["fp16", "fp16", "fp16", "fp32", "fp16_h2"])
        layout = rng.choice(["internal", "canonical"])
        additive = rng.random() < 0.15
        nrhs = rng.choice([1, 1, 2, 5]) if layout == "internal" and volume(c) <= 700000 else 1
        i_s = rng.choice([1, 2, 4, 16]) if volume(c) <= 200000 else rng.choice([1, 2, 4])
        return dict(c, kind=kind, prec=prec, layout=layout, nrhs=nrhs, i_s=i_s, i_d=rng.randint(2, 6), additive=additive)
    if kind == "setup":
        return dict(draw_lattice(rng, 24 ** 3 * 48), kind=kind)
    c = draw_lattice(rng, 24 ** 3 * 48)
    m = rng.choice([12, 16, 24, 32])
    i_s = rng.choice([2, 4, 8])
    return dict(c, kind=kind, prec=rng.choice(["fp16", "fp16", "fp32"]), nrhs=rng.choice([1, 1, 2, 3]), i_s=i_s,
                i_d=rng.choice([3, 4, 5]), m=m, k=rng.choice([0, 4, 6]), steps=100 // i_s)


# ------------------------------------------------------------------ sizes
def dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def domain(case):
    return case["bx"], case["by"], case["bz"], case["bt"]


def volume(case):
    return math.prod(dims(case))


def apply_work(case, prec, nrhs):
    """Four links and the clover blocks (72 reals each) once, 24 reals in and 24 out per
    right-hand side; 1848 flop per site (eight hops of 168 and the clover's 504)."""
    v = volume(case)
    norms = 8 if prec == "fp16" else 0
    return v * (144 * REAL_BYTES[prec] + nrhs * (48 * REAL_BYTES[prec] + norms)), 1848 * v * nrhs


def sap_work(case, prec, i_s, i_d, nrhs):
    """Matrices once, FP32 fields in and out; per site and visit I_d minimal-residual steps
    (hops inside the domain, clover or its inverse, inner products and updates), one more
    half of each for the preparation and for the reconstruction, and the faces."""
    v = volume(case)
    inside = sum(2.0 * (b - 1) / b for b in domain(case))
    face = 8.0 - inside
    visit = (i_d + 1) * (168 * inside + 504) + i_d * 192 + 48 + face * 168
    return v * (144 * REAL_BYTES[prec] + nrhs * 192), i_s * visit * v * nrhs


def work(case):
    v = volume(case)
    if case["kind"] == "apply":
        b, f = apply_work(case, case["prec"], case["nrhs"])
    elif case["kind"] == "sap":
        b, f = sap_work(case, case["prec"], case["i_s"], case["i_d"], case["nrhs"])
    elif case["kind"] == "setup":
        # the links once; the six planes' leaves (ten 3x3 products each) and two 6x6 inverses;
        # then one FP64 operator and one single-precision preconditioner application
        ba, fa = apply_work(case, "fp64", 1)
        bs, fs = sap_work(case, "fp32", 1, 4, 1)
        b, f = v * 72 * 8 + ba + bs, v * (6 * 10 * 198 + 2 * 8 * 6 ** 3 / 3) + fa + fs
    else:
        # `steps` Arnoldi steps per source: M, A, the projection of step j against the j + 1
        # vectors before it (two passes), and the FP64 residual at the end
        n, s = case["nrhs"], case["steps"]
        b1, f1 = sap_work(case, case["prec"], case["i_s"], case["i_d"], n)
        b2, f2 = apply_work(case, "fp32", n)
        b3, f3 = apply_work(case, "fp64", n)
        mean = min(s, case["m"]) / 2 + 1
        b, f = s * (b1 + b2 + n * v * 96 * 2 * mean) + b3, s * (f1 + f2 + n * v * 192 * mean) + f3
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    """About four times the distance from exact() seen on the listed lattices."""
    if case["kind"] == "apply":
        return {"rel": {"fp64": 5e-16, "fp32": 3.5e-7, "fp16": 1.5e-3}[case["prec"]]}
    if case["kind"] == "sap":
        return {"rel": {"fp32": 6e-7, "fp16": 2e-3, "fp16_h2": 4.5e-3}[case["prec"]]}
    if case["kind"] == "setup":
        return {"rel": 6e-7}
    # |f - A x| <= 1e-10 |f| is all that a solve promises: up to 1e-9 was seen in x
    return {"rel": 5e-9}


# ------------------------------------------------------------------ inputs
# Site fields below are component first, [..., T, Z, Y, X]: every operation is elementwise on
# contiguous planes.  Direction mu = 0..3 (x, y, z, t) is axis -1 - mu.
def mm(a, b):
    """3x3 products of [3, 3, ...] fields."""
    return sum(a[:, k, None] * b[None, k] for k in range(3))


def dag(a):
    return a.transpose(0, 1).conj()


def unitary(m):
    """SU(3) by Gram-Schmidt on the rows."""
    r0 = m[0] / m[0].abs().square().sum(0).sqrt()
    r1 = m[1] - (r0.conj() * m[1]).sum(0) * r0
    r1 = r1 / r1.abs().square().sum(0).sqrt()
    r2 = torch.stack([r0[1] * r1[2] - r0[2] * r1[1], r0[2] * r1[0] - r0[0] * r1[2], r0[0] * r1[1] - r0[1] * r1[0]]).conj()
    return torch.stack([r0, r1, r2])


def gauge(case, gen):
    """Four [3, 3, T, Z, Y, X] link fields: exp(i width H), H a Gaussian Hermitian traceless
    matrix, then `smear` steps of APE smearing (alpha = 1/2)."""
    shape = dims(case)[::-1]
    links = []
    for _ in range(4):
        e = torch.randn((8,) + shape, generator=gen, device="cuda", dtype=torch.float64) * (0.5 * case["width"])
        z, d = torch.zeros_like(e[0]), e[7] / math.sqrt(3)
        re = torch.stack([e[2] + d, e[0], e[3], e[0], d - e[2], e[5], e[3], e[5], -2 * d])
        im = torch.stack([z, -e[1], -e[4], e[1], z, -e[6], e[4], e[6], z])
        h = torch.complex(-im, re).reshape((3, 3) + shape) / 4  # i H / 4
        one = torch.eye(3, device="cuda", dtype=h.dtype).reshape(3, 3, 1, 1, 1, 1)
        x = one + h / 14
        for n in range(13, 0, -1):
            x = one + mm(h, x) / n
        x = mm(x, x)
        links.append(unitary(mm(x, x)))
    for _ in range(case["smear"]):
        new = []
        for mu in range(4):
            s = 0
            for nu in range(4):
                if nu != mu:
                    n, m = links[nu], links[mu]
                    s = s + mm(mm(n, m.roll(-1, -1 - nu)), dag(n.roll(-1, -1 - mu)))
                    nb = n.roll(1, -1 - nu)
                    s = s + mm(mm(dag(nb), m.roll(1, -1 - nu)), nb.roll(-1, -1 - mu))
            new.append(unitary(0.5 * links[mu] + s / 12))
        links = new
    return links


def sources(case, gen):
    """nrhs Gaussian spinor fields [4, 3, T, Z, Y, X]."""
    shape = (4, 3) + dims(case)[::-1]
    r = [torch.randn(shape + (2,), generator=gen, device="cuda", dtype=torch.float64) for _ in range(case.get("nrhs", 1))]
    return [torch.view_as_complex(v) for v in r]


def inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return gauge(case, gen), sources(case, gen)


def canonical(psi):
    """[4, 3, T, Z, Y, X] complex -> the library's [t, z, y, x, spin, colour, re/im]."""
    return torch.view_as_real(psi.permute(2, 3, 4, 5, 0, 1).contiguous())


def internal(psi, case):
    """[4, 3, T, Z, Y, X] complex -> the library's domain-major field: per domain six units of
    four reals, each over the even, then the odd sites of the domain."""
    (bx, by, bz, bt), (lx, ly, lz, lt) = domain(case), dims(case)
    v = canonical(psi).reshape(lt // bt, bt, lz // bz, bz, ly // by, by, lx // bx, bx, 24)
    v = v.permute(0, 2, 4, 6, 1, 3, 5, 7, 8).reshape(-1, bx * by * bz * bt, 6, 4)
    t, z, y, x = (torch.arange(b, device="cuda") for b in (bt, bz, by, bx))
    parity = (t[:, None, None, None] + z[:, None, None] + y[:, None] + x).reshape(-1) % 2
    order = torch.argsort(parity, stable=True)
    return v[:, order].permute(0, 2, 1, 3).contiguous()


def arrange(fields, case, layout):
    return torch.stack([canonical(f) if layout == "canonical" else internal(f, case) for f in fields])


def prepare(case, seed):
    links, src = inputs(case, seed)
    shape = dims(case)[::-1]
    field = torch.view_as_real(torch.stack(links).permute(3, 4, 5, 6, 0, 1, 2).contiguous())
    ctx = dd.Context(dims(case), domain(case), True, torch.cuda.current_stream().cuda_stream)
    state = {"case": dict(case), "ctx": ctx}
    if case["kind"] == "setup":
        state["links"] = field
        state["in64"] = canonical(src[0])
        state["in32"] = state["in64"].float()
        state["out64"], state["out32"] = torch.empty_like(state["in64"]), torch.empty_like(state["in32"])
        torch.cuda.synchronize()
        return state
    torch.cuda.synchronize()
    ctx.dd_load_gauge(field, dd.DD_DEVICE)
    ctx.dd_build_clover(case["kappa"], case["csw"])
    del field, links
    if case["kind"] == "solve":
        state["f"] = arrange(src, case, "canonical")
        state["x"] = torch.empty_like(state["f"])
    elif case["prec"] == "fp16" and case["kind"] == "apply":
        each = ctx.dd_spinor_bytes(dd.DD_PREC_FP16, dd.DD_LAYOUT_INTERNAL)
        state["in"] = torch.empty((len(src), each), dtype=torch.uint8, device="cuda")
        state["half"] = torch.empty_like(state["in"])
        for f, buf in zip(src, state["in"]):
            f32 = canonical(f).float()
            torch.cuda.synchronize()
            ctx.dd_pack_spinor(f32, dd.DD_PREC_FP32, buf, dd.DD_PREC_FP16)
        state["out"] = torch.empty((len(src),) + shape + (4, 3, 2), dtype=torch.float32, device="cuda")
    else:
        state["in"] = arrange(src, case, case["layout"]).to(torch.float64 if case["prec"] == "fp64" else torch.float32)
        state["out"] = torch.empty_like(state["in"])
    torch.cuda.synchronize()
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "apply":
        prec = PREC[case["prec"]]
        where = dd.DD_LAYOUT_CANONICAL if case["layout"] == "canonical" else dd.DD_LAYOUT_INTERNAL
        out = state["half"] if case["prec"] == "fp16" else state["out"]
        if case["nrhs"] > 1:
            ctx.dd_apply_D_batch(state["in"], out, case["nrhs"], prec)
        else:
            ctx.dd_apply_D(state["in"], out, prec, where)
        if case["prec"] == "fp16":  # half fields are read back in single precision
            for h, o in zip(state["half"], state["out"]):
                ctx.dd_unpack_spinor(h, prec, o, dd.DD_PREC_FP32)
        return state["out"]
    if case["kind"] == "sap":
        args = (case["i_s"], case["i_d"], PREC[case["prec"]])
        if case["nrhs"] > 1:
            ctx.dd_sap_precondition_batch(state["in"], state["out"], case["nrhs"], *args, additive=int(case["additive"]))
        else:
            where = dd.DD_LAYOUT_CANONICAL if case["layout"] == "canonical" else dd.DD_LAYOUT_INTERNAL
            ctx.dd_sap_precondition(state["in"], state["out"], *args, where, additive=int(case["additive"]))
        return state["out"]
    if case["kind"] == "setup":
        ctx.dd_load_gauge(state["links"], dd.DD_DEVICE)
        ctx.dd_build_clover(case["kappa"], case["csw"])
        ctx.dd_apply_D(state["in64"], state["out64"], dd.DD_PREC_FP64)
        ctx.dd_sap_precondition(state["in32"], state["out32"], 1, 4, dd.DD_PREC_FP32)
        return {"residual": state["out64"], "preconditioned": state["out32"]}
    state["x"].zero_()
    ctx.dd_solve(state["f"], state["x"], nrhs=case["nrhs"], where=dd.DD_DEVICE, tol=1e-10, m=case["m"], k=case["k"],
                 max_iter=4000, i_schwarz=case["i_s"], i_domain=case["i_d"], storage_prec=PREC[case["prec"]])
    return state["x"]


# ------------------------------------------------------------------ the same in FP64, plain torch
# gamma_k = [[0, -i s_k], [i s_k, 0]], gamma_t = [[0, 1], [1, 0]]: gamma_mu psi as (source spin,
# factor) for each of the four spins
GAMMA = [[(3, -1j), (2, -1j), (1, 1j), (0, 1j)], [(3, -1), (2, 1), (1, 1), (0, -1)],
         [(2, -1j), (3, 1j), (0, 1j), (1, -1j)], [(2, 1), (3, 1), (0, 1), (1, 1)]]


class Operator:
    """A = 1/(2 kappa) - D_w / 2 + D_cl, antiperiodic in t, and its restriction to domains."""

    def __init__(self, case, links):
        self.case, self.axes = case, [-1, -2, -3, -4]
        self.clover = self.build_clover(links, case)
        links = [u for u in links]
        last = links[3].clone()
        last[:, :, -1] *= -1  # the fermion's boundary condition, folded into the last time slice
        links[3] = last
        self.fwd = links
        self.bwd = [dag(u.roll(1, -1 - mu)).contiguous() for mu, u in enumerate(links)]
        pos = torch.meshgrid(*[torch.arange(n, device="cuda") for n in dims(case)[::-1]], indexing="ij")[::-1]
        self.odd = sum(pos) % 2 == 1
        dom = [p // b for p, b in zip(pos, domain(case))]
        self.white = sum(dom) % 2 == 1
        self.in_fwd = [p % b != b - 1 for p, b in zip(pos, domain(case))]
        self.in_bwd = [p % b != 0 for p, b in zip(pos, domain(case))]

    @staticmethod
    def build_clover(links, case):
        f = {}
        for mu in range(4):
            for nu in range(mu + 1, 4):
                m, n, am, an = links[mu], links[nu], -1 - mu, -1 - nu
                up = mm(mm(m, n.roll(-1, am)), mm(dag(m.roll(-1, an)), dag(n)))  # the plaquette at x
                left = mm(mm(n, dag(m.roll(-1, an).roll(1, am))), mm(dag(n.roll(1, am)), m.roll(1, am)))
                nd, md = n.roll(1, am).roll(1, an), m.roll(1, am).roll(1, an)
                down = mm(mm(dag(m.roll(1, am)), dag(nd)), mm(md, n.roll(1, an)))
                right = mm(mm(dag(n.roll(1, an)), m.roll(1, an)), mm(n.roll(1, an).roll(-1, am), dag(m)))
                q = up + left + down + right
                f[mu, nu] = q - dag(q)
        # -(c_sw / 32) sum_{mu != nu} gamma_mu gamma_nu F_mu,nu, block diagonal in chirality
        out = torch.zeros((2, 6, 6) + dims(case)[::-1], dtype=torch.complex128, device="cuda")
        for (mu, nu), fm in f.items():
            for s in range(4):
                k, a = GAMMA[mu][s]
                t, b = GAMMA[nu][k]
                i, j = 3 * (s % 2), 3 * (t % 2)
                out[s // 2, i:i + 3, j:j + 3] += (-case["csw"] / 16 * a * b) * fm
        for i in range(6):
            out[:, i, i] += 1 / (2 * case["kappa"])
        return out

    def hops(self, psi, inside):
        """sum over mu of the forward and backward hops (those inside the domains only)."""
        out = torch.zeros_like(psi)
        for mu in range(4):
            for sign, u, step, keep in ((-1, self.fwd[mu], -1, self.in_fwd[mu]), (1, self.bwd[mu], 1, self.in_bwd[mu])):
                p = psi.roll(step, -1 - mu)
                if inside:
                    p = p * keep
                h = torch.stack([p[s] + sign * GAMMA[mu][s][1] * p[GAMMA[mu][s][0]] for s in (0, 1)])
                h = u[:, 0] * h[:, 0, None] + u[:, 1] * h[:, 1, None] + u[:, 2] * h[:, 2, None]
                out[:2] += h
                for s in (2, 3):
                    k, a = GAMMA[mu][s]
                    out[s] += sign * a * h[k]
        return out

    @staticmethod
    def blocks(c, psi):
        v = psi.reshape((2, 6) + psi.shape[2:])
        y = c[:, :, 0] * v[:, 0, None]
        for j in range(1, 6):
            y += c[:, :, j] * v[:, j, None]
        return y.reshape(psi.shape)

    def apply(self, psi):
        return self.blocks(self.clover, psi) - 0.5 * self.hops(psi, False)

    def schwarz(self, f, i_s, i_d, additive):
        """I_S Schwarz iterations; each domain is solved by I_d minimal-residual steps on the
        even sites' Schur complement."""
        c = self.clover.permute(3, 4, 5, 6, 0, 1, 2).contiguous()
        inv = torch.linalg.inv(c).permute(4, 5, 6, 0, 1, 2, 3).contiguous()
        (bx, by, bz, bt), (lx, ly, lz, lt) = domain(self.case), dims(self.case)
        split = (lt // bt, bt, lz // bz, bz, ly // by, by, lx // bx, bx)

        def dot(a, b):  # per domain, spread over its sites
            s = (a.conj() * b).sum((0, 1)).reshape(split).sum((1, 3, 5, 7), keepdim=True)
            return s.expand(split).reshape(lt, lz, ly, lx)

        u = torch.zeros_like(f)
        for _ in range(i_s):
            for colour in ((None,) if additive else (False, True)):
                r = f - self.apply(u)
                mine = torch.ones_like(self.odd) if colour is None else self.white == colour
                r = r * mine
                ro = r * self.odd
                e = (r + 0.5 * self.hops(self.blocks(inv, ro), True)) * ~self.odd
                x = torch.zeros_like(f)
                for _ in range(i_d):
                    t = self.blocks(inv, self.hops(e, True) * self.odd)
                    p = (self.blocks(self.clover, e) - 0.25 * self.hops(t, True)) * ~self.odd
                    a, n = dot(p, e), dot(p, p).real
                    a = torch.where(n > 0, a / torch.where(n > 0, n, 1), 0)
                    x = x + a * e
                    e = e - a * p
                u = u + (x + self.blocks(inv, (ro + 0.5 * self.hops(x, True)) * self.odd)) * mine
        return u

    def solve(self, f):
        """BiCGstab to a true residual below 1e-12."""
        x, r = torch.zeros_like(f), f.clone()
        norm = f.abs().square().sum().sqrt()
        vdot = lambda a, b: torch.vdot(a.reshape(-1), b.reshape(-1))
        for _ in range(4):
            shadow, p = r.clone(), r.clone()
            rho = vdot(shadow, r)
            for k in range(2000):
                v = self.apply(p)
                alpha = rho / vdot(shadow, v)
                r -= alpha * v
                t = self.apply(r)
                omega = vdot(t, r) / vdot(t, t)
                x += alpha * p + omega * r
                r -= omega * t
                new = vdot(shadow, r)
                p = r + (new / rho * alpha / omega) * (p - omega * v)
                rho = new
                if k % 8 == 7 and r.abs().square().sum().sqrt() < 1e-13 * norm:
                    break
            r = f - self.apply(x)
            if r.abs().square().sum().sqrt() < 1e-12 * norm:
                break
        return x


def exact(case, seed):
    links, src = inputs(case, seed)
    op = Operator(case, links)
    del links
    if case["kind"] == "apply":
        layout = "canonical" if case["prec"] == "fp16" else case["layout"]
        return arrange([op.apply(f) for f in src], case, layout)
    if case["kind"] == "sap":
        return arrange([op.schwarz(f, case["i_s"], case["i_d"], case["additive"]) for f in src], case, case["layout"])
    if case["kind"] == "setup":
        return {"residual": canonical(op.apply(src[0])), "preconditioned": canonical(op.schwarz(src[0], 1, 4, False))}
    return arrange([op.solve(f) for f in src], case, "canonical")
