"""The work a user of this library has it do, as cases that can be timed: single calls of the
public binding (`paper_1501_01855_gb300.binding.Overlap`) on synthetic gauge fields.

The lattices are those of the repository's configurations, tests and benchmark (4^4, 8^4,
8^3 x 16, 16^3 x 32, 24^3 x 48) and ragged ones in between; links are smooth random SU(3)
(proj_SU3 of 1 + i eps H + (i eps H)^2 / 2, eps = 0.3), sources Gaussian or point sources,
m0 = 1.4, 20 Zolotarev poles on [0.2, 2.6] as in the benchmark. A context (the gauge field in
the library's layouts, Zolotarev data) and, where one is used, a deflation space are what a
user's program holds before the call; every pass is one call on device tensors.

Kinds: "apply" D(mu) v (or gamma5 D(mu) v, or the sign alone), "wilson" K v, "solve" the
inverter, "gram" a Gram block, "ritz" one Ritz step, "force" the gauge-link gradient.
"""
import math

import numpy as np
import torch

from paper_1501_01855_gb300 import binding as B

M0 = 1.4
KAPPA = 1.0 / (8.0 - 2.0 * M0)
POLES = 20
LOW, HIGH = 0.2, 2.6
PRECS = {"f64": B.OVL_PREC_F64, "f32": B.OVL_PREC_F32, "f64e": B.OVL_PREC_F64E, "auto": B.OVL_PREC_AUTO}


def listed():
    return [
        # the smallest call: one vector on the lattice of the first configuration; all latency
        dict(name="apply_4x4x4x4_n1", kind="apply", lx=4, ly=4, lz=4, lt=4, n=1, eta=1e-10, prec="auto", c64=False,
             op="D", mu=0.05, apt=False),
        # gamma5 D on a few vectors of a small test lattice, antiperiodic in t (the usual fermion boundary)
        dict(name="apply_8x8x8x16_n4", kind="apply", lx=8, ly=8, lz=8, lt=16, n=4, eta=1e-10, prec="auto", c64=False,
             op="H", mu=0.05, apt=True),
        # the headline: D(mu) to 1e-10 on 16^3 x 32, a vector for each of the 12 spin-colour sources
        dict(name="apply_16x16x16x32_n12", kind="apply", lx=16, ly=16, lz=16, lt=32, n=12, eta=1e-10, prec="auto",
             c64=False, op="D", mu=0.05, apt=False),
        # the single-precision sign of a batch of 12 spin-colour sources, the inner work of every relaxed solve
        dict(name="sign_f32_16x16x16x32_n12", kind="apply", lx=16, ly=16, lz=16, lt=32, n=12, eta=1e-6, prec="f32",
             c64=True, op="sign", mu=0.05, apt=False),
        # one vector on a ragged lattice (sites not a multiple of any block), loose accuracy
        dict(name="sign_f32_10x6x14x12_n1", kind="apply", lx=10, ly=6, lz=14, lt=12, n=1, eta=1e-4, prec="f32",
             c64=True, op="sign", mu=0.05, apt=True),
        # K alone on the largest configured lattice, single precision
        dict(name="wilson_f32_24x24x24x48_n1", kind="wilson", lx=24, ly=24, lz=24, lt=48, n=1, prec="f32", c64=True,
             apt=False),
        # K of 12 vectors in FP64
        dict(name="wilson_f64_16x16x16x32_n12", kind="wilson", lx=16, ly=16, lz=16, lt=32, n=12, prec="f64", c64=False,
             apt=False),
        # one right-hand side by the mixed-precision inverter (GMRESR(relSUMR))
        dict(name="solve_16x16x16x32_n1", kind="solve", lx=16, ly=16, lz=16, lt=32, n=1, masses=1, mu=0.05, cg=False,
             half=False, n_ev=0, tol=1e-11),
        # 12 point sources at three masses in one batch, deflated by 16 eigSUMR vectors
        dict(name="solve_defl_8x8x8x16_n12x3", kind="solve", lx=8, ly=8, lz=8, lt=16, n=12, masses=3, mu=0.05, cg=False,
             half=False, n_ev=16, tol=1e-11),
        # the dense block of a Ritz step at basis size 128
        dict(name="gram_f64_16x16x16x32_128x128", kind="gram", lx=16, ly=16, lz=16, lt=32, na=128, nb=128, g5=False,
             c64=False),
        # one whole Ritz step (Gram blocks, host algebra, rotation), 64 vectors to 16
        dict(name="ritz_8x8x8x32_64to16", kind="ritz", lx=8, ly=8, lz=8, lt=32, m=64, keep=16, mu=0.05),
        # the fermion force of the gradient configuration in plain FP64 (two inversions, every pole's shifted systems)
        dict(name="force_8x8x8x8", kind="force", lx=8, ly=8, lz=8, lt=8, mu=0.05, mixed=False, tol=1e-12),
    ]


def _dims(rng, lo, hi):
    """Even extents with a volume of about exp(uniform(log lo, log hi)) sites."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        d = [rng.choice((4, 6, 8, 10, 12, 14, 16)) for _ in range(3)] + [rng.choice((4, 6, 8, 10, 12, 16, 20, 24, 32))]
        v = d[0] * d[1] * d[2] * d[3]
        if 0.6 * want <= v <= min(hi, 1.5 * want):
            return dict(lx=d[0], ly=d[1], lz=d[2], lt=d[3])


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "wilson", "wilson", "solve", "gram", "ritz", "force"))
    if kind == "apply":
        f32 = rng.random() < 0.4
        return dict(kind=kind, **_dims(rng, 256, 131072), n=_log_int(rng, 1, 12), mu=rng.choice((0.02, 0.05, 0.2)),
                    eta=rng.choice((1e-4, 1e-6)) if f32 else rng.choice((1e-8, 1e-10)), prec="f32" if f32 else "auto",
                    c64=f32, op=rng.choice(("D", "H", "sign")), apt=rng.random() < 0.5)
    if kind == "wilson":
        f32 = rng.random() < 0.5
        return dict(kind=kind, **_dims(rng, 256, 131072), n=_log_int(rng, 1, 16),
                    prec="f32" if f32 else rng.choice(("f64", "f64e")), c64=f32, apt=rng.random() < 0.5)
    if kind == "solve":
        return dict(kind=kind, **_dims(rng, 256, 8192), n=_log_int(rng, 1, 6), masses=rng.choice((1, 1, 2, 3)),
                    mu=rng.choice((0.05, 0.1, 0.2)), cg=rng.random() < 0.3, half=rng.random() < 0.3, n_ev=0, tol=1e-11)
    if kind == "gram":
        return dict(kind=kind, **_dims(rng, 256, 32768), na=_log_int(rng, 1, 192), nb=_log_int(rng, 1, 192),
                    g5=rng.random() < 0.5, c64=rng.random() < 0.3)
    if kind == "ritz":
        m = _log_int(rng, 8, 128)
        return dict(kind=kind, **_dims(rng, 512, 16384), m=m, keep=max(1, m // rng.choice((2, 3, 4, 6))), mu=0.05)
    return dict(kind=kind, **_dims(rng, 256, 4096), mu=rng.choice((0.05, 0.1)), mixed=False, tol=1e-12)


# ---------------------------------------------------------------- inputs
def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _sites(case):
    return (case["lt"], case["lz"], case["ly"], case["lx"])


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _links(case, seed):
    """Smooth random SU(3) links [t][z][y][x][mu][3][3], complex128, on the GPU."""
    h = torch.randn(_sites(case) + (4, 8), generator=_generator(seed, 1), device="cuda", dtype=torch.float64) * 0.5
    H = torch.zeros(h.shape[:-1] + (3, 3), device="cuda", dtype=torch.complex128)
    for (i, j), re, im in (((0, 1), 0, 1), ((0, 2), 3, 4), ((1, 2), 5, 6)):
        H[..., i, j] = torch.complex(h[..., re], -h[..., im])
        H[..., j, i] = torch.complex(h[..., re], h[..., im])
    s = h[..., 7] / math.sqrt(3.0)
    H[..., 0, 0], H[..., 1, 1], H[..., 2, 2] = (h[..., 2] + s).to(H.dtype), (s - h[..., 2]).to(H.dtype), (-2 * s).to(H.dtype)
    H *= 0.3j
    m = torch.eye(3, device="cuda", dtype=torch.complex128) + H + 0.5 * (H @ H)
    r1 = m[..., 0, :] / torch.linalg.vector_norm(m[..., 0, :], dim=-1, keepdim=True)
    r2 = m[..., 1, :] - (r1.conj() * m[..., 1, :]).sum(-1, keepdim=True) * r1
    r2 = r2 / torch.linalg.vector_norm(r2, dim=-1, keepdim=True)
    return torch.stack((r1, r2, torch.linalg.cross(r1, r2).conj()), dim=-2)


def _vectors(case, seed, n, stream=2):
    """n Gaussian spinors [n][t][z][y][x][4][3] of the case's element type."""
    dt = torch.complex64 if case.get("c64") else torch.complex128
    return math.sqrt(2.0) * torch.randn((n,) + _sites(case) + (4, 3), generator=_generator(seed, stream), device="cuda",
                                        dtype=dt)


def _point_sources(case, seed, n):
    """Spin-colour point sources at a site of the seed's (one Gaussian source instead when n = 1)."""
    if n == 1:
        return _vectors(case, seed, 1)
    at = np.random.default_rng(int(seed)).integers(0, _volume(case))
    b = torch.zeros((n, _volume(case), 12), device="cuda", dtype=torch.complex128)
    for j in range(n):
        b[j, at, j % 12] = 1.0
    return b.view((n,) + _sites(case) + (4, 3))


def _masses(case):
    return [case["mu"] * (1 + k) for k in range(case.get("masses", 1))]


def _context(case, seed, links=None):
    p = B.ovl_params_default()
    p.a_override, p.b_override = LOW, HIGH
    p.bc_t = 1 if case.get("apt") else 0
    p.mixed = 1 if case.get("mixed", True) else 0
    p.half_storage = 1 if case.get("half") else 0
    p.solver = B.OVL_SOLVER_CG if case.get("cg") else B.OVL_SOLVER_SUMR
    U = _links(case, seed) if links is None else links
    dims = (case["lx"], case["ly"], case["lz"], case["lt"])
    return B.Overlap(dims, U.cpu().numpy(), M0, case.get("mu", 0.05), POLES, 1e-10, params=p)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "ctx": _context(case, seed)}
    if kind in ("apply", "wilson"):
        s["v"] = _vectors(case, seed, case["n"])
        s["out"] = torch.empty_like(s["v"])
    elif kind == "solve":
        s["b"] = _point_sources(case, seed, case["n"])
        s["x"] = torch.empty((case["masses"] * case["n"],) + s["b"].shape[1:], dtype=s["b"].dtype, device="cuda")
        s["defl"] = None
        if case["n_ev"]:
            b0 = _vectors(case, seed, 1, stream=3)
            s["defl"], _ = s["ctx"].eigsumr_accumulate(b0, torch.empty_like(b0), 1e-10, case["n_ev"], 3 * case["n_ev"])
    elif kind == "gram":
        s["A"], s["B"] = _vectors(case, seed, case["na"]), _vectors(case, seed, case["nb"], stream=3)
    elif kind == "ritz":
        s["v"] = _vectors(case, seed, case["m"])
        s["v"] /= math.sqrt(24.0 * _volume(case))
        s["vD"] = s["ctx"].apply(s["v"], torch.empty_like(s["v"]), eta=1e-8)
    else:
        s["phi"] = _vectors(case, seed, 1)
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "apply":
        if case["op"] == "sign":
            return ctx.sign_apply(s["v"], s["out"], eta=case["eta"], prec=PRECS[case["prec"]])
        return ctx.apply(s["v"], s["out"], eta=case["eta"], prec=PRECS[case["prec"]], hermitian=case["op"] == "H")
    if kind == "wilson":
        return ctx.wilson_apply(s["v"], s["out"], prec=PRECS[case["prec"]])
    if kind == "solve":
        ctx.solve(s["b"], s["x"], case["tol"], mus=_masses(case), defl=s["defl"])
        return s["x"]
    if kind == "gram":
        return ctx.gram(s["A"], s["B"], g5=1 if case["g5"] else 0,
                        prec=B.OVL_PREC_F32 if case["c64"] else B.OVL_PREC_F64)
    if kind == "ritz":
        ritz, v, vD, res = ctx.ritz_recalculate(s["v"], s["vD"], case["keep"])
        return {"ritz": ritz, "v": v, "vD": vD, "res": res}
    G, S = ctx.force(s["phi"], tol=case["tol"])
    return {"G": G, "S": S}


# ---------------------------------------------------------------- what a pass cannot do without
def _krylov_steps(eta):
    """Steps of the Krylov space of K^2 to a sign of accuracy eta (the CG bound on [LOW, HIGH])."""
    return 0.5 * (HIGH / LOW) * math.log(2.0 / eta)


def work(case):
    V, kind = _volume(case), case["kind"]
    spinor = 12 * V * (8 if case.get("c64") else 16)
    links = 4 * V * 12 * (4 if case.get("c64") else 8)
    hop = 1368.0 * V
    if kind == "wilson":
        return {"bytes": 2 * case["n"] * spinor + links, "flops": case["n"] * hop}
    if kind == "apply":
        return {"bytes": 2 * case["n"] * spinor + links, "flops": case["n"] * hop * (2 * _krylov_steps(case["eta"]) + 1)}
    if kind == "gram":
        return {"bytes": (case["na"] + case["nb"]) * spinor, "flops": 8.0 * case["na"] * case["nb"] * 12 * V}
    if kind == "ritz":
        m, k = case["m"], case["keep"]
        return {"bytes": (2 * m + 2 * k) * spinor, "flops": (3 * 8.0 * m * m + 2 * 8.0 * m * k) * 12 * V}
    # an inversion: about 2 / mu ln(1 / tol) Krylov steps, the sign in each relaxed to half the digits on average
    signs = 0.5 / case["mu"] * math.log(2.0 / case["tol"])
    one = hop * signs * 2 * _krylov_steps(math.sqrt(case["tol"]))
    if kind == "solve":
        n = case["n"] * case["masses"]
        return {"bytes": (case["n"] + n) * spinor + links, "flops": n * one}
    return {"bytes": spinor + links + 36 * V * 16, "flops": 2 * one + 4 * hop * _krylov_steps(case["tol"])}


# ---------------------------------------------------------------- 64-bit values
def _gammas():
    i, z = 1j, 0
    g = np.array([[[z, z, z, i], [z, z, i, z], [z, -i, z, z], [-i, z, z, z]],
                  [[z, z, z, -1], [z, z, 1, z], [z, 1, z, z], [-1, z, z, z]],
                  [[z, z, i, z], [z, z, z, -i], [-i, z, z, z], [z, i, z, z]],
                  [[z, z, 1, z], [z, z, z, 1], [1, z, z, z], [z, 1, z, z]]], dtype=np.complex128)
    return torch.from_numpy(g).cuda()


class _Plain:
    """K and the sign function in plain torch, complex128; fields as [t][z][y][x][colour][spin x n]."""

    def __init__(self, case, seed):
        self.case, self.U, self.gam = case, _links(case, seed), _gammas()
        self.Ud = self.U.conj().transpose(-1, -2).contiguous()
        self.n = 0

    def pack(self, v):
        self.n = v.shape[0]
        return v.to(torch.complex128).permute(1, 2, 3, 4, 6, 5, 0).reshape(_sites(self.case) + (3, 4 * self.n)).contiguous()

    def unpack(self, p):
        return p.view(_sites(self.case) + (3, 4, self.n)).permute(6, 0, 1, 2, 3, 5, 4).contiguous()

    def g5(self, p):
        q = p.clone()
        q[..., 2 * self.n:] *= -1
        return q

    def _gamma(self, mu, p):
        q = p.view(p.shape[:-1] + (4, self.n))
        return torch.matmul(self.gam[mu], q).view(p.shape)

    def K(self, p):
        hop = torch.zeros_like(p)
        for mu in range(4):
            ax = 3 - mu
            f = torch.roll(p, -1, ax)
            if mu == 3 and self.case.get("apt"):
                f[-1] *= -1
            f = torch.matmul(self.U[..., mu, :, :], f)
            hop += f - self._gamma(mu, f)
            b = torch.matmul(self.Ud[..., mu, :, :], p)
            b = torch.roll(b, 1, ax)
            if mu == 3 and self.case.get("apt"):
                b[0] *= -1
            hop += b + self._gamma(mu, b)
        return self.g5(p - KAPPA * hop)

    def sign(self, p):
        """sign(K) p: K times the Chebyshev series of s^(-1/2) in s = K^2 on an interval that covers the spectrum."""
        lo, hi, deg = 0.15 ** 2, 2.7 ** 2, 300
        N = 4 * deg
        th = (np.arange(N) + 0.5) * math.pi / N
        fx = (0.5 * (hi + lo) + 0.5 * (hi - lo) * np.cos(th)) ** -0.5
        c = np.array([2.0 / N * np.sum(fx * np.cos(k * th)) for k in range(deg + 1)])
        c[0] *= 0.5
        a, b0 = 2.0 / (hi - lo), (hi + lo) / (hi - lo)
        T0, T1 = p, a * self.K(self.K(p)) - b0 * p
        y = c[0] * T0 + c[1] * T1
        for k in range(2, deg + 1):
            T2 = 2.0 * a * self.K(self.K(T1)) - 2.0 * b0 * T1 - T0
            y += c[k] * T2
            T0, T1 = T1, T2
        return self.K(y)


def exact(case, seed):
    kind = case["kind"]
    if kind == "wilson":
        P = _Plain(case, seed)
        return P.unpack(P.K(P.pack(_vectors(case, seed, case["n"]))))
    if kind == "apply":
        P = _Plain(case, seed)
        v = P.pack(_vectors(case, seed, case["n"]))
        s = P.sign(v)
        if case["op"] == "D":
            s = 0.5 * (1 + case["mu"]) * v + 0.5 * (1 - case["mu"]) * P.g5(s)
        elif case["op"] == "H":
            s = 0.5 * (1 + case["mu"]) * P.g5(v) + 0.5 * (1 - case["mu"]) * s
        return P.unpack(s)
    if kind == "gram":
        A = _vectors(case, seed, case["na"]).flatten(1).to(torch.complex128)
        b = _vectors(case, seed, case["nb"], stream=3).to(torch.complex128)
        if case["g5"]:
            b[..., 2:, :] *= -1
        return torch.matmul(A.conj(), b.flatten(1).transpose(0, 1))
    return None   # solutions, eigenvectors up to a phase, and the gradient have no such quick plain form
