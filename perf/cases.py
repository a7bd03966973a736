"""What this library's users have it do, as cases that can be timed and checked.

A case is one call of a public entry point: the operator on vectors, shifted solves on device arrays,
FS-MLMC level traces (plain, Wilson-clover, probed and diluted with the hopping parameter expansion)
and variance sampling. Lattices, shifts, masses, levels, displacements and precisions are those of the
benchmark's, the tests' and the serving workload's configurations. Fields are synthetic: Haar or
smoothed SU(3) links, Gaussian vectors, the library's own Z4 noise.

Mixed-precision solves run to 1e-11 and FP64 ones to 1e-12, what a correlator-grade inversion (and the
tests against dense inverses) asks: the results are then fixed by the problem, not by the path of the
iteration. Solver statistics (iteration counts) belong to that path and are not outputs.
"""

import math

import numpy as np
import torch

import paper_2212_04430_gb300 as fs
from paper_2212_04430_gb300.fsmlmc import wilson_dslash_noalloc

TOL = {"f64": 1e-12, "f32": 1e-11, "f16": 1e-11, "bf16": 1e-11}
SERVE_LATTICES = ((8, 8, 8, 8), (8, 8, 8, 16), (12, 12, 12, 24), (16, 16, 16, 32))


def _case(name, kind, dims, **kw):
    c = {"name": name, "kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "bc": -1,
         "links": "smooth", "eps": 0.3, "m": -0.2, "csw": 0.0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: (D + sigma) on one host vector, a residual check on a test lattice
        _case("dslash_4x4_f64", "dslash", (4, 4, 4, 4), prec="f64", link=18, nrhs=1, s0=0.15, nlev=1, ds=1.0,
              links="haar", m=-0.4),
        # the allocation-free operator on device arrays: twelve spin-colour components on 8^4
        _case("dslash_dev_8x8_f64", "dslash_dev", (8, 8, 8, 8), prec="f64", link=18, nrhs=12, s0=0.1, nlev=1, ds=1.0),
        # the 4^4 Haar job: two shifts, Gamma = 1, p = 0, 64 Z4 vectors per level, FP64
        _case("mlmc_4x4_f64", "mlmc", (4, 4, 4, 4), prec="f64", link=18, tile=32, s0=0.0, nlev=2, ds=0.4, nvec=64,
              gamma="I", p=0, est="diff", links="haar", m=-0.4),
        # shifted solves of a few caller vectors on device arrays, library-chosen tile, FP32 storage
        _case("solve_8x8_f32", "solve", (8, 8, 8, 8), prec="f32", link=18, tile=0, s0=0.02, nlev=3, ds=0.2, nrhs=5),
        # the 8^4 job: three levels, gamma5 gamma3, p = 2, FP32 storage, 16-system tiles
        _case("mlmc_8x8_f32", "mlmc", (8, 8, 8, 8), prec="f32", link=18, tile=16, s0=0.02, nlev=3, ds=0.24, nvec=32,
              gamma="g5g3", p=2, est="split_even"),
        # one job of the serving mix on 8^3x16: four levels, FP16 storage, 32-system tiles
        _case("mlmc_8x16_f16", "mlmc", (8, 8, 8, 16), prec="f16", link=18, tile=32, s0=0.01, nlev=4, ds=0.2, nvec=32,
              gamma="g5g4", p=3, est="split_even"),
        # the paper's noise on a small lattice: 16 probing colours, full spin-colour dilution and the
        # hopping parameter expansion of the last level, one sample per level
        _case("probed_4x8_f16", "probed", (4, 4, 4, 8), prec="f16", link=12, tile=32, s0=0.05, nlev=2, ds=0.55, nvec=1,
              gamma="g3", p=2, est="split_even", hpe=4),
        # a ragged lattice, an odd number of right-hand sides, BF16 storage, a tile that fits neither
        _case("solve_ragged_bf16", "solve", (6, 10, 14, 12), prec="bf16", link=18, tile=12, s0=0.03, nlev=3, ds=0.15,
              nrhs=7),
        # few right-hand sides on the benchmark lattice: two shifts of four vectors, FP16 storage
        _case("solve_16x32_f16", "solve", (16, 16, 16, 32), prec="f16", link=12, tile=8, s0=0.03, nlev=2, ds=0.57,
              nrhs=4, m=-0.35, eps=0.4),
        # Wilson-clover level traces on a lattice whose sides are not powers of two
        _case("clover_12x24_f16", "mlmc", (12, 12, 12, 24), prec="f16", link=12, tile=32, s0=0.01, nlev=4, ds=0.2,
              nvec=8, gamma="g3", p=4, est="split_even", csw=1.0),
        # the benchmark job: 16^3x32, four levels, gamma3, p = 4, FP16 storage, 12-real links,
        # 32-system tiles
        _case("mlmc_16x32_f16", "mlmc", (16, 16, 16, 32), prec="f16", link=12, tile=32, s0=0.005, nlev=4, ds=0.198,
              nvec=16, gamma="g3", p=4, est="split_even", m=-0.35, eps=0.4),
        # variance sampling at 24^3x64: five sampling shifts, every displacement 0..8
        _case("varsample_24x64_f16", "varsample", (24, 24, 24, 64), prec="f16", link=12, tile=32, s0=0.0, nlev=5, ds=0.25,
              nvec=2, gamma="g3", p=8, hpe=0, m=-0.38, eps=0.5),
    ]


def _dims_near(rng, v, least=(2, 2, 2, 2)):
    """Four even sides with a volume near v, none of them special."""
    side = v ** 0.25
    d = [max(least[k], 2 * round(side * rng.uniform(0.7, 1.4) / 2)) for k in range(3)]
    d.append(max(least[3], 2 * round(v / (d[0] * d[1] * d[2]) / 2)))
    return tuple(int(x) for x in d)


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("dslash", "dslash_dev", "solve", "solve", "mlmc", "mlmc", "mlmc", "probed", "varsample"))
    kw = dict(bc=rng.choice((-1, -1, -1, 1)), links="smooth", eps=round(rng.uniform(0.3, 0.4), 3),
              m=round(rng.uniform(-0.25, -0.1), 3), s0=round(_log(rng, 0.01, 0.1), 4), ds=round(rng.uniform(0.1, 0.4), 3),
              csw=0.0, nlev=1)
    gam, est = rng.choice(("I", "g3", "g5g3", "g5g4", "g5")), rng.choice(("split_even", "split_even", "diff", "product"))
    low = rng.choice(("f16", "f16", "f16", "bf16", "f32"))
    if kind == "dslash":
        prec = rng.choice(("f64", "f64", "f32"))
        kw.update(prec=prec, link=18 if prec == "f64" else rng.choice((12, 18)), nrhs=rng.choice((1, 1, 2, 5, 12, 17)))
        dims = _dims_near(rng, _log(rng, 64, 3e5 / kw["nrhs"]))
    elif kind == "dslash_dev":
        kw.update(prec="f64", link=18, nrhs=rng.choice((1, 3, 4, 12, 20)))
        dims = _dims_near(rng, _log(rng, 64, 0.55 * (2 ** 25) / (576 + 384 * kw["nrhs"])))
    elif kind == "solve":
        prec = rng.choice((low, low, "f64"))
        kw.update(prec=prec, link=18 if prec == "f64" else rng.choice((12, 18)), nlev=rng.choice((1, 2, 3, 5)),
                  nrhs=rng.choice((1, 2, 3, 7, 12)), tile=rng.choice((0, 4, 12, 24, 32)))
        if kw["nlev"] * kw["nrhs"] >= 16 and kw["tile"] == 0:
            kw["tile"] = 32
        dims = _dims_near(rng, _log(rng, 128, (3e5 if prec == "f64" else 2e6) / (kw["nlev"] * kw["nrhs"])))
    elif kind == "varsample":
        kw.update(prec=low, link=rng.choice((12, 18)), tile=rng.choice((20, 32, 64)), nlev=rng.choice((3, 5)),
                  nvec=rng.choice((1, 2, 5)), gamma=gam, p=rng.choice((0, 2, 4)), hpe=rng.choice((0, 0, 4)))
        dims = _dims_near(rng, _log(rng, 1024, 2e6 / (2 * kw["nlev"] * kw["nvec"])), (2, 2, 6, 2))
    elif kind == "probed":
        kw.update(prec=rng.choice((low, "f64")), link=18, tile=rng.choice((16, 32, 60)), nlev=rng.choice((1, 2)), nvec=1,
                  gamma=gam, p=rng.choice((0, 1, 2)), est="split_even", hpe=rng.choice((0, 2, 4)))
        dims = _dims_near(rng, _log(rng, 256, 900 if kw["hpe"] or kw["prec"] == "f64" else 3000), (4, 4, 4, 4))
    else:
        prec = rng.choice((low, low, low, "f64"))
        kw.update(prec=prec, link=18 if prec == "f64" else rng.choice((12, 18)), tile=rng.choice((8, 16, 32, 32, 48, 64)),
                  nlev=rng.choice((1, 2, 3, 4, 6)), gamma=gam, p=rng.choice((0, 1, 2, 3, 4)), est=est,
                  csw=rng.choice((0.0, 0.0, 1.0)))
        if prec != "f64" and rng.random() < 0.4:
            dims = rng.choice(SERVE_LATTICES[:3])
        else:
            dims = _dims_near(rng, _log(rng, 256, 4096 if prec == "f64" else 50000), (2, 2, 6, 2))
        v = dims[0] * dims[1] * dims[2] * dims[3]
        most = (2e5 if prec == "f64" else 3e6) / (v * (2 * kw["nlev"] - 1))
        kw["nvec"] = max(1, min(64, int(_log(rng, 4, max(5.0, most)))))
    c = _case("", kind, dims, **kw)
    del c["name"]
    return c


# ---- inputs -------------------------------------------------------------------------------------

def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _sigmas(case):
    return [case["s0"] + k * case["ds"] for k in range(case["nlev"])]


def _gaussian(g, shape):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, device="cuda", dtype=torch.float64)) / math.sqrt(2)


def _links(case, seed):
    """Links complex128 [4][V][3][3] on the GPU: Haar (Gram-Schmidt of a Gaussian matrix) or exp(i eps H)."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1))
    a = _gaussian(g, (4 * _volume(case), 3, 3))
    if case["links"] == "haar":
        r0 = a[:, 0] / torch.linalg.vector_norm(a[:, 0], dim=-1, keepdim=True)
        r1 = a[:, 1] - (r0.conj() * a[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        u = torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], 1)
    else:
        h = 0.5 * (a + a.mH)
        eye = torch.eye(3, dtype=h.dtype, device="cuda")
        h = h - (torch.einsum("nii->n", h) / 3.0)[:, None, None] * eye
        x = (1j * case["eps"] / 16.0) * h  # exp by its series on x / 16, then four squarings
        u = eye + x / 12.0
        for k in range(11, 0, -1):
            u = eye + (x @ u) / k
        for _ in range(4):
            u = u @ u
    return u.reshape(4, _volume(case), 3, 3)


def _vectors(case, seed):
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + 1)
    return _gaussian(g, (case["nrhs"], _volume(case), 4, 3))


def _noise_seed(seed):
    return 2000 + 7919 * (seed + 1)


def _site(case):
    x = np.arange(_volume(case))
    lx, ly, lz, _ = _dims(case)
    return x % lx, x // lx % ly, x // (lx * ly) % lz, x // (lx * ly * lz)


def _colors(case):
    """Hierarchical probing's first 16 colours: the parity of each coordinate."""
    x, y, z, t = _site(case)
    return ((x & 1) + 2 * (y & 1) + 4 * (z & 1) + 8 * (t & 1)).astype(np.int32)


def prepare(case, seed):
    """What a user's program keeps: a context with its gauge field, the vectors, the noise's seed."""
    u = _links(case, seed)
    s = {"case": case, "sigma": _sigmas(case), "seed": _noise_seed(seed)}
    if case["kind"] == "dslash_dev":
        s["u"] = torch.view_as_real(u).contiguous()
        s["in"] = torch.view_as_real(_vectors(case, seed)).contiguous()
        s["out"] = torch.empty_like(s["in"])
        s["stream"] = torch.cuda.current_stream().cuda_stream
        return s
    s["ctx"] = fs.Context(_dims(case), bc_t=case["bc"], device=0)
    s["ctx"].fs_set_gauge(u.cpu().numpy())
    if case["csw"]:
        s["ctx"].fs_set_clover(case["csw"])
    if case["kind"] == "dslash":
        s["in"] = _vectors(case, seed).cpu().numpy()
    elif case["kind"] == "solve":
        s["in"] = torch.view_as_real(_vectors(case, seed)).contiguous()
        s["out"] = torch.empty((case["nlev"],) + tuple(s["in"].shape), dtype=torch.float64, device="cuda")
    else:
        s["gamma"] = fs.gamma_matrix(case["gamma"])
        s["colors"] = _colors(case) if case["kind"] == "probed" else None
    torch.cuda.synchronize()
    return s


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "dslash":
        return state["ctx"].wilson_dslash(c["m"], c["s0"], state["in"], prec=c["prec"], link_compress=c["link"])
    if kind == "dslash_dev":
        rc = wilson_dslash_noalloc(_dims(c), c["bc"], c["m"], c["s0"], state["u"].data_ptr(), state["in"].data_ptr(),
                                   state["out"].data_ptr(), c["nrhs"], state["stream"])
        if rc:
            raise RuntimeError("wilson_dslash_noalloc: status %d" % rc)
        return state["out"]
    kw = dict(prec=c["prec"], link_compress=c["link"], tol=TOL[c["prec"]], rhs_tile=c["tile"])
    if kind == "solve":
        state["ctx"].shifted_solve_dev(c["m"], state["sigma"], state["in"].data_ptr(), c["nrhs"], state["out"].data_ptr(),
                                       **kw)
        return state["out"]
    if kind == "varsample":
        r = state["ctx"].variance_sample(c["m"], state["sigma"], state["gamma"], list(range(c["p"] + 1)), c["nvec"],
                                         seed=state["seed"], hpe_order=c["hpe"], **kw)
        return {k: r[k] for k in ("a", "b", "VL", "Vbar")}
    if kind == "probed":
        kw.update(colors=state["colors"], ncolors=16, dilute=True, hpe_order=c["hpe"])
    r = state["ctx"].mlmc_level_trace(c["m"], state["sigma"], state["gamma"], c["p"], [c["nvec"]] * c["nlev"],
                                      seed=state["seed"], estimator=c["est"], **kw)
    return {"samples": np.concatenate(r["samples"]), "trace": r["trace"], "var": r["var"]}


def _solves(case):
    if case["kind"] == "solve":
        return case["nlev"] * case["nrhs"]
    if case["kind"] == "varsample":
        return 2 * case["nlev"] * case["nvec"]
    return (2 * case["nlev"] - 1) * case["nvec"] * (192 if case["kind"] == "probed" else 1)


def work(case):
    """Links and vectors once; the operator's 1320 flop per site (1368 with the diagonal) once, or, for a solve, in each of
    two applications of 40 iterations (a nominal count: the shifts and masses here take 20 to 120)."""
    v = _volume(case)
    if case["kind"] in ("dslash", "dslash_dev"):
        return {"bytes": v * (576.0 + 384.0 * case["nrhs"]), "flops": 1368.0 * v * case["nrhs"]}
    n = _solves(case)
    vec = 192.0 * v * (case["nrhs"] * (1 + case["nlev"])) if case["kind"] == "solve" else 0.0
    return {"bytes": 576.0 * v + vec, "flops": 80.0 * 1368.0 * v * n}


# ---- the same values in 64 bits, in plain torch --------------------------------------------------
# Vectors are complex128 [Lt][Lz][Ly][Lx][colour 3][spin 4][n], links [4][Lt][Lz][Ly][Lx][3][3].

_I = 1j
_G = (((0, _I), (_I, 0)), ((0, -1), (1, 0)), ((_I, 0), (0, -_I)), ((1, 0), (0, 1)))  # gamma_mu = [[0, G], [G^dag, 0]]


def _gammas():
    out = []
    for g in _G:
        m = np.zeros((4, 4), complex)
        m[:2, 2:] = np.array(g)
        m[2:, :2] = np.array(g).conj().T
        out.append(m)
    return out


def _t(a):
    return torch.as_tensor(np.asarray(a, dtype=complex), dtype=torch.complex128, device="cuda")


def _axis(mu):
    return 3 - mu


class _Exact:
    def __init__(self, case, seed):
        self.case = case
        self.shape = (case["lt"], case["lz"], case["ly"], case["lx"])
        self.u = _links(case, seed).reshape((4,) + self.shape + (3, 3))
        self.udag = [torch.roll(self.u[mu], 1, _axis(mu)).mH.contiguous() for mu in range(4)]
        ub = [self.u[mu].clone() for mu in range(4)]
        ub[3][-1] *= case["bc"]
        self.ubc = ub
        db = [d.clone() for d in self.udag]
        db[3][0] *= case["bc"]
        self.dbc = db
        self.gam = _gammas()
        self.minus = [_t(np.eye(4) - g) for g in self.gam]
        self.plus = [_t(np.eye(4) + g) for g in self.gam]
        self.clover = self._clover(case["csw"]) if case["csw"] else None

    def mul(self, u, psi):  # colour
        return (u.reshape(-1, 3, 3) @ psi.reshape(psi.shape[:4].numel(), 3, -1)).reshape(psi.shape)

    def spin(self, g, psi):
        return torch.einsum("st,zyxwctn->zyxwcsn", g, psi)

    def hop(self, psi):
        """H psi, D = 4 + m - H / 2."""
        out = torch.zeros_like(psi)
        for mu in range(4):
            ax = _axis(mu)
            out += self.spin(self.minus[mu], self.mul(self.ubc[mu], torch.roll(psi, -1, ax)))
            out += self.spin(self.plus[mu], self.mul(self.dbc[mu], torch.roll(psi, 1, ax)))
        return out

    def _clover(self, csw):
        def sh(a, mu, n):  # a(x + n mu)
            return torch.roll(a, -n, _axis(mu))
        v = int(np.prod(self.shape))
        c = torch.zeros((v, 3, 4, 3, 4), dtype=torch.complex128, device="cuda")
        for mu in range(4):
            for nu in range(mu + 1, 4):
                um, un = self.u[mu], self.u[nu]
                q = um @ sh(un, mu, 1) @ sh(um, nu, 1).mH @ un.mH
                q = q + un @ sh(sh(um, nu, 1), mu, -1).mH @ sh(un, mu, -1).mH @ sh(um, mu, -1)
                q = q + sh(um, mu, -1).mH @ sh(sh(un, mu, -1), nu, -1).mH @ sh(sh(um, mu, -1), nu, -1) @ sh(un, nu, -1)
                q = q + sh(un, nu, -1).mH @ sh(um, nu, -1) @ sh(sh(un, mu, 1), nu, -1) @ um.mH
                f = ((q - q.mH) / 8j).reshape(v, 3, 3)
                s = 0.5j * (self.gam[mu] @ self.gam[nu] - self.gam[nu] @ self.gam[mu])
                c += torch.einsum("st,vab->vasbt", _t(0.5 * csw * s), f)
        return c.reshape(v, 12, 12)

    def cterm(self, psi):
        return (self.clover @ psi.reshape(self.clover.shape[0], 12, -1)).reshape(psi.shape)

    def apply(self, sig, psi):
        out = (4.0 + self.case["m"] + sig) * psi - 0.5 * self.hop(psi)
        return out + self.cterm(psi) if self.clover is not None else out

    def solve(self, sig, b):
        """(D + sig_j)^-1 b_j by BiCGStab, restarted from the true residual until that stops falling."""
        x, n2 = torch.zeros_like(b), self.norm2(b)
        last = None
        for _ in range(8):
            r = b - self.apply(sig, x)
            worst = float((self.norm2(r) / n2).max()) ** 0.5
            if worst < 1e-14 or (last is not None and worst > 0.3 * last):
                break
            last = worst
            x = x + self.correction(sig, r)
        return x

    def norm2(self, a):
        return a.real.square().sum((0, 1, 2, 3, 4, 5)) + a.imag.square().sum((0, 1, 2, 3, 4, 5))

    def dot(self, a, b):
        return (a.conj() * b).sum((0, 1, 2, 3, 4, 5))

    def correction(self, sig, b):
        x, r, p = torch.zeros_like(b), b.clone(), b.clone()
        rh, rho, goal = b.clone(), self.dot(b, b), self.norm2(b) * 1e-16
        live = torch.ones_like(goal)
        for k in range(3000):
            v = self.apply(sig, p)
            al = torch.nan_to_num(rho / self.dot(rh, v)) * live
            s = r - al * v
            t = self.apply(sig, s)
            om = torch.nan_to_num(self.dot(t, s) / self.norm2(t)) * live
            x = x + al * p + om * s
            r = s - om * t
            rho2 = self.dot(rh, r)
            be = torch.nan_to_num((rho2 / rho) * (al / om)) * live
            p = torch.where(live > 0, r + be * (p - om * v), p)
            rho = torch.where(live > 0, rho2, rho)
            live = (self.norm2(r) > goal).double()
            if k % 8 == 7 and not bool(live.any()):
                break
        return x

    def omega(self, p, psi):
        """(Omega_p psi)(x) = U_z(x) ... U_z(x + (p-1) z) psi(x + p z)."""
        for _ in range(p):
            psi = self.mul(self.u[2], torch.roll(psi, -1, _axis(2)))
        return psi

    def insert(self, left, gamma, p, psi):
        return self.dot(left, self.spin(gamma, self.omega(p, psi)))


def _philox(case, sample, level, job, seed):
    """Philox4x32-10 word 0 of every site, and from it z = i^k as [V][4 spin][3 colour]."""
    m32 = np.uint64(0xFFFFFFFF)
    v = _volume(case)
    c = [np.arange(v, dtype=np.uint64)] + [np.full(v, w & 0xFFFFFFFF, np.uint64) for w in (sample, level, job)]
    k = [seed & 0xFFFFFFFF, seed >> 32]
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        s = np.uint64(32)
        c = [(b >> s) ^ c[1] ^ np.uint64(k[0]), b & m32, (a >> s) ^ c[3] ^ np.uint64(k[1]), a & m32]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    code = (c[0][:, None] >> np.arange(0, 24, 2, dtype=np.uint64)[None, :]) & np.uint64(3)
    return np.array([1, 1j, -1, -1j])[code.astype(int)].reshape(v, 4, 3)


def _fields(e, vecs):
    """[n][V][spin][colour] -> the layout of _Exact."""
    a = vecs if torch.is_tensor(vecs) else _t(vecs)
    return a.permute(1, 3, 2, 0).reshape(e.shape + (3, 4, a.shape[0])).contiguous()


def _vecs(psi):
    """Back: [n][V][spin][colour]."""
    n = psi.shape[-1]
    return psi.reshape(-1, 3, 4, n).permute(3, 0, 2, 1).contiguous()


def _var(c):
    return float(np.mean(np.abs(c - c.mean()) ** 2))


def _gamma(name):
    g = _gammas()
    m = np.eye(4, dtype=complex)
    while name not in ("", "I"):
        m = m @ (np.diag([1, 1, -1, -1]).astype(complex) if name[1] == "5" else g[int(name[1]) - 1])
        name = name[2:]
    return _t(m)


def _expansion(e, case, sig, k, psi):
    """(kappa H)^k psi, kappa H = H / (2 A); Wilson."""
    for _ in range(k):
        psi = e.hop(psi) / (2.0 * (4.0 + case["m"] + sig))
    return psi


def _low_orders(e, case, gamma, sig):
    """sum_{k < K} Tr(Gamma Omega_p (kappa H)^k) / A from every unit vector."""
    v, total = _volume(case), 0.0
    step = max(12, (1 << 24) // (12 * v) // 12 * 12)
    for lo in range(0, 12 * v, step):
        n = min(step, 12 * v - lo)
        z = torch.zeros(12 * v, n, dtype=torch.complex128, device="cuda")
        z[torch.arange(lo, lo + n), torch.arange(n)] = 1.0
        z = z.reshape(e.shape + (3, 4, n))
        y = z
        for k in range(case["hpe"]):
            total += complex(e.insert(z, gamma, case["p"], y).sum().item())
            y = _expansion(e, case, sig, 1, y)
    return total / (4.0 + case["m"] + sig)


def _g5(psi):
    out = psi.clone()
    out[..., 2:, :] *= -1
    return out


def exact(case, seed):
    v, kind = _volume(case), case["kind"]
    if kind not in ("dslash", "dslash_dev") and v * _solves(case) > 3.2e6:
        return None
    e, sig = _Exact(case, seed), _sigmas(case)
    if kind in ("dslash", "dslash_dev"):
        out = _vecs(e.apply(case["s0"], _fields(e, _vectors(case, seed))))
        return out.cpu().numpy() if kind == "dslash" else torch.view_as_real(out)
    if kind == "solve":
        b = _fields(e, _vectors(case, seed))
        return torch.stack([torch.view_as_real(_vecs(e.solve(s, b))) for s in sig])
    gamma, key = _gamma(case["gamma"]), _noise_seed(seed)
    if kind == "varsample":
        z = _fields(e, np.stack([_philox(case, k, 0x80000000, 0, key) for k in range(case["nvec"])]))
        x = [e.solve(s, z) for s in sig]
        y = [_g5(e.solve(s, _g5(z))) for s in sig]
        n, ps = len(sig), range(case["p"] + 1)
        a, b = np.zeros((case["nvec"], len(ps), n), complex), np.zeros((case["nvec"], len(ps), n, n), complex)
        for i in range(n):
            xr = _expansion(e, case, sig[i], case["hpe"], x[i]) if case["m"] + sig[i] > 0 else x[i]
            for p in ps:
                a[:, p, i] = e.insert(z, gamma, p, xr).cpu().numpy()
                for j in range(i, n):
                    b[:, p, i, j] = e.insert(y[i], gamma, p, x[j]).cpu().numpy()
        return {"a": a, "b": b, "VL": np.array([[_var(a[:, p, i]) for i in range(n)] for p in ps]),
                "Vbar": np.array([[[_var(b[:, p, i, j]) for j in range(n)] for i in range(n)] for p in ps])}
    expand = kind == "probed" and case["hpe"] > 0 and case["m"] + sig[-1] > 0
    if expand and v > 1024:
        return None
    samples = []
    for lev in range(case["nlev"]):
        pieces = []
        for k in range(case["nvec"]):
            z = _philox(case, k, lev, 0, key)
            if kind == "probed":
                col = _colors(case)
                for c in range(16):
                    for comp in range(12):
                        q = np.zeros_like(z)
                        q[col == c, comp // 3, comp % 3] = z[col == c, comp // 3, comp % 3]
                        pieces.append(q)
            else:
                pieces.append(z)
        z = _fields(e, np.stack(pieces))
        if lev + 1 == case["nlev"]:
            x = e.solve(sig[lev], z)
            val = e.insert(z, gamma, case["p"], _expansion(e, case, sig[lev], case["hpe"], x) if expand else x)
        elif case["est"] == "split_even":
            y = _g5(e.solve(sig[lev], _g5(z)))
            val = (sig[lev + 1] - sig[lev]) * e.insert(y, gamma, case["p"], e.solve(sig[lev + 1], z))
        else:  # difference and product agree sample by sample
            val = e.insert(z, gamma, case["p"], e.solve(sig[lev], z) - e.solve(sig[lev + 1], z))
        val = val.reshape(case["nvec"], -1).sum(1).cpu().numpy()
        if expand and lev + 1 == case["nlev"]:
            val = val + _low_orders(e, case, gamma, sig[lev])
        samples.append(val)
    return {"samples": np.concatenate(samples), "trace": np.array([s.mean() for s in samples]),
            "var": np.array([_var(s) for s in samples])}
