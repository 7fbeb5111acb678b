"""What is measured: the calls that a program using this library makes.

A case is one call (or the call sequence of one gauge configuration) through
the binding of the C ABI, on torch CUDA tensors and the current stream:

    dslash    one operator application (tm_dslash)
    gauge     a new configuration: link upload, packing and check
              (tsm_load_gauge), then one application of D_tm on it
    solve     D_tm s = b for a batch of Z4 sources (tm_solve_batch)
    tsm       a whole TSM estimate (tsm_loops): the loops, their error and the
              LP mean
    contract  the loops of one given solution (tsm_contract)
    net       forward pass of the learned preconditioner (tsm_net_forward)

Sizes are those of the library's workloads (4^4, 8^3x16, 12^3x24, 16^3x32,
24^3x48) and, in draw(), everything between them with extents such as 6, 10,
14 or 22 and odd source counts.  Truncated (LP) solves run a fixed number of
iterations (tm_stop.rel_tol = 0, the rule that the paper treats as
interchangeable with a residual; 8 is what 5e-3 takes on these fields), so
that every source's work is the same on every machine.

The ABI hands every result back as doubles, whatever the tier computed.  run()
narrows each result to the type its tier computes in, as a program that stores
it does: complex128 for FP64 (and the reliable-update solves), complex64 for
FP32, 16-bit reals for the results of 16-bit solves (loops per site of a
timeslice, so that they fit the range).  Diagnostics that rounding decides
(residual norms, iteration counts of a tolerance) are not results.
"""
import math

import torch

from paper_1211_0126_gb300 import tsm

KAPPA, MU, EPS = 0.1245, 0.005, 0.25
GAMMAS = list(range(16))
F64, F32, BF16, F16 = tsm.TSM_F64, tsm.TSM_F32, tsm.TSM_BF16, tsm.TSM_F16
HP_TOL, HP_DELTA = 1e-10, 1e-5     # the high-precision stop inside tsm_loops
SOLVE_TOL = 1e-12                  # and of a high-precision solve whose solution is kept
OPS = {"full": tsm.TM_OP_FULL, "schur": tsm.TM_OP_SCHUR, "normal": tsm.TM_OP_NORMAL}
REAL_BYTES = {F64: 8, F32: 4, BF16: 2, F16: 2}


def _case(name, kind, dims, **kw):
    return dict({"name": name, "kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3]}, **kw)


def listed():
    return [
        # an operator on the smallest lattice (unit tests, dense checks): launches and host work count
        _case("dslash-f64-4x4x4x4", "dslash", (4, 4, 4, 4), prec=F64, op="full"),
        # the preconditioned operator in FP32, as a caller's own Krylov method applies it
        _case("dslash-f32-16x16x16x32", "dslash", (16, 16, 16, 32), prec=F32, op="schur"),
        # the full operator in the LP tier at production size
        _case("dslash-f16-24x24x24x48", "dslash", (24, 24, 24, 48), prec=F16, op="full"),
        # the next configuration of an ensemble
        _case("gauge-24x24x24x48", "gauge", (24, 24, 24, 48), prec=F32),
        # a batch of truncated solves
        _case("solve-f16-16x16x16x32", "solve", (16, 16, 16, 32), prec=F16, nrhs=32, iters=8),
        # a batch of high-precision solves (FP32 iterations, FP64 reliable updates)
        _case("solve-hp-12x12x12x24", "solve", (12, 12, 12, 24), prec=F32, nrhs=8, iters=0),
        # the production estimate: 8 HP and 256 LP sources, 16 insertions at 7 momenta
        _case("tsm-24x24x24x48", "tsm", (24, 24, 24, 48), prec=F16, iters=8, n_hp=8, n_lp=256, batch=32, nq=7,
              deriv=0, fft=False),
        # the small lattice of the batching workload, BF16 tier
        _case("tsm-bf16-8x8x8x16", "tsm", (8, 8, 8, 16), prec=BF16, iters=7, n_hp=8, n_lp=64, batch=64, nq=7,
              deriv=0, fft=False),
        # local and one-derivative insertions along x, y, z, t at 13 momenta
        _case("tsm-deriv-12x12x12x24", "tsm", (12, 12, 12, 24), prec=F16, iters=8, n_hp=4, n_lp=32, batch=16, nq=13,
              deriv=15, fft=False),
        # every spatial momentum through the FFT projection
        _case("tsm-fft-16x16x16x32", "tsm", (16, 16, 16, 32), prec=F16, iters=8, n_hp=2, n_lp=32, batch=32, nq=1,
              deriv=0, fft=True),
        # the loops of one stored solution
        _case("contract-f32-24x24x24x48", "contract", (24, 24, 24, 48), prec=F32, nq=7),
        # one application of the learned preconditioner's network
        _case("net-16x16x16x32", "net", (16, 16, 16, 32), nb=1, hidden=12, layers=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, vmin, vmax):
    """Even extents with a volume spread over [vmin, vmax] on a log scale."""
    while True:
        v = _log(rng, vmin, vmax)
        s = (v / 2.0) ** 0.25
        d = [max(4, 2 * round(s * _log(rng, 0.75, 1.34) / 2)) for _ in range(3)]
        t = max(4, 2 * round(v / (d[0] * d[1] * d[2]) / 2))
        if t <= 64 and d[0] * d[1] * d[2] * t <= vmax and all(_smooth(x) for x in d):
            return d + [t]


def _smooth(n):
    for p in (2, 3, 5, 7, 11, 13):
        while n % p == 0:
            n //= p
    return n == 1


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "gauge", "solve", "solve", "tsm", "tsm", "contract", "net"])
    big, mid, small = 24 ** 3 * 48, 16 ** 3 * 32, 12 ** 3 * 24
    if kind == "dslash":
        c = _case("", kind, _dims(rng, 256, big), prec=rng.choice([F64, F32, F16, BF16]),
                  op=rng.choice(["full", "schur", "normal"]))
    elif kind == "gauge":
        c = _case("", kind, _dims(rng, 4096, big), prec=rng.choice([F32, F16]))
    elif kind == "solve":
        if rng.random() < 0.6:
            c = _case("", kind, _dims(rng, 2048, mid), prec=F16, nrhs=int(_log(rng, 4, 33)), iters=rng.randint(5, 10))
        else:
            c = _case("", kind, _dims(rng, 2048, small), prec=F32, nrhs=rng.randint(2, 12), iters=0)
    elif kind == "tsm":
        form = rng.choice(["plain", "plain", "deriv", "fft"])
        c = _case("", kind, _dims(rng, 2048, mid if form == "plain" else small),
                  prec=rng.choice([F16, F16, BF16]), iters=rng.randint(5, 9), n_hp=rng.randint(2, 8),
                  n_lp=int(_log(rng, 8, 97)), batch=int(_log(rng, 4, 33)),
                  nq=1 if form == "fft" else rng.choice([1, 4, 7, 13]),
                  deriv=rng.choice([4, 7, 15]) if form == "deriv" else 0, fft=form == "fft")
        if form == "fft":
            c["prec"] = F16
    elif kind == "contract":
        c = _case("", kind, _dims(rng, 256, big), prec=rng.choice([F32, F32, F64]), nq=rng.choice([1, 4, 7, 13]))
    else:
        c = _case("", kind, _dims(rng, 512, mid), nb=1, hidden=rng.choice([12, 16, 24]) if rng.random() < 0.5 else 12,
                  layers=rng.choice([2, 3]))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _dims_of(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(1000003 * (seed % (1 << 40)) + salt)


def _normal(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), dtype=torch.float64, device="cuda", generator=gen))


def _matmul3(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _links(dims, seed):
    """SU(3) links exp(i EPS H), H a random traceless hermitian matrix: [T, Z, Y, X, 4, 3, 3]."""
    lx, ly, lz, lt = dims
    gen = _gen(seed, 1)
    a = _normal((lt, lz, ly, lx, 4, 3, 3), gen)
    h = 0.5 * (a + a.mH)
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    x = (1j * EPS / 8) * (h - (h.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3) * eye)
    out, term = eye + x, x
    for k in range(2, 8):
        term = _matmul3(term, x) / k
        out = out + term
    for _ in range(3):
        out = _matmul3(out, out)
    r1 = out[..., 0, :]
    r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
    r2 = out[..., 1, :]
    r2 = r2 - (r1.conj() * r2).sum(-1, keepdim=True) * r1
    r2 = r2 / r2.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack([r1, r2, torch.linalg.cross(r1, r2).conj()], dim=-2).resolve_conj().contiguous()


def _spinors(c, seed, n=None):
    lx, ly, lz, lt = _dims_of(c)
    return _normal(((n,) if n else ()) + (lt, lz, ly, lx, 4, 3), _gen(seed, 2))


def _z4(c, seed):
    lx, ly, lz, lt = _dims_of(c)
    bits = torch.randint(0, 2, (c["nrhs"], lt, lz, ly, lx, 4, 3, 2), device="cuda", generator=_gen(seed, 3))
    return torch.view_as_complex((bits.to(torch.float64) * 2 - 1) / math.sqrt(2.0))


def _channels(c):
    return [1] + [c["hidden"]] * (c["layers"] - 1) + [1]


def _weights(c, seed):
    """Near-identity weights as a trained network has: [4 C_out, 36 C_in] per layer."""
    gen, ch, out = _gen(seed, 4), _channels(c), []
    for ci, co in zip(ch[:-1], ch[1:]):
        w = _normal((4 * co, 36 * ci), gen) * (0.3 / math.sqrt(36 * ci))
        for o in range(co):
            for s in range(4):
                for i in range(ci) if co == 1 else [o % ci]:
                    w[4 * o + s, 4 * i + s] += 1.0 / ci if co == 1 else 1.0
        out.append(w.to(torch.complex64).to(torch.complex128))
    return out


def _hp_stop(tol):
    return tsm.stop(tol, 20000, F32, reliable=True, reliable_delta=HP_DELTA)


def prepare(case, seed):
    dims, kind = _dims_of(case), case["kind"]
    ctx = tsm.Context(0, torch.cuda.current_stream().cuda_stream)
    links = _links(dims, seed)
    st = {"case": case, "ctx": ctx, "dims": dims, "kind": kind}
    if kind == "gauge":
        st["links"], st["psi"] = links, _spinors(case, seed)
        st["out"] = torch.empty_like(st["psi"])
        return st
    ctx.load_gauge(links, dims, KAPPA, MU)
    if kind == "dslash":
        st["psi"] = _spinors(case, seed)
        st["out"] = torch.empty_like(st["psi"])
    elif kind == "solve":
        st["b"] = _z4(case, seed)
        st["s"] = torch.empty_like(st["b"])
        st["stop"] = tsm.stop(0.0, case["iters"], case["prec"]) if case["iters"] else _hp_stop(SOLVE_TOL)
    elif kind == "tsm":
        moms = _momenta(case["nq"])
        n_hp, n_lp = case["n_hp"], case["n_lp"]
        st["params"] = tsm.params(seed, 4, (0, n_hp), (n_hp, n_hp + n_lp), _hp_stop(HP_TOL),
                                  tsm.stop(0.0, case["iters"], case["prec"]), GAMMAS, moms, batch=case["batch"],
                                  deriv_mask=case["deriv"], all_momenta=case["fft"])
        lx, ly, lz, lt = dims
        shape = (16, lt, lz, ly, lx) if case["fft"] else (16, len(moms), lt)
        if case["deriv"]:
            shape = (1 + bin(case["deriv"]).count("1"),) + shape
        st["loops"] = torch.empty(shape, dtype=torch.complex128, device="cuda")
        st["mean"] = torch.empty_like(st["loops"])
        st["err"] = torch.empty(shape, dtype=torch.float64, device="cuda")
    elif kind == "contract":
        st["s"], st["seed"] = _spinors(case, seed), seed
        st["moms"] = _momenta(case["nq"])
        st["out"] = torch.empty((16, len(st["moms"]), dims[3]), dtype=torch.complex128, device="cuda")
    else:
        st["net"] = tsm.Network(_channels(case))
        for l, w in enumerate(_weights(case, seed)):
            st["net"].set_weights(l, w.cpu().numpy())
        st["x"] = _spinors(case, seed, 1)[:, None].contiguous()
        st["y"] = torch.empty_like(st["x"])
    return st


# ------------------------------------------------------------------ one pass
def _narrow(x, prec):
    if prec == F64:
        return x
    if prec == F32:
        return x.to(torch.complex64 if x.is_complex() else torch.float32)
    return (torch.view_as_real(x) if x.is_complex() else x).to(torch.float16)


def run(st):
    c, ctx, kind = st["case"], st["ctx"], st["kind"]
    if kind == "dslash":
        tsm.tm_dslash(ctx.h, c["prec"], OPS[c["op"]], False, st["psi"], st["out"])
        return _narrow(st["out"], c["prec"])
    if kind == "gauge":
        ctx.load_gauge(st["links"], st["dims"], KAPPA, MU)
        tsm.tm_dslash(ctx.h, c["prec"], tsm.TM_OP_FULL, False, st["psi"], st["out"])
        return _narrow(st["out"], c["prec"])
    if kind == "solve":
        tsm.tm_solve_batch(ctx.h, st["b"], st["s"], st["stop"], c["nrhs"])
        return _narrow(st["s"], c["prec"] if c["iters"] else F64)
    if kind == "tsm":
        tsm.tsm_loops(ctx.h, st["params"], st["loops"], st["err"], st["mean"])
        return _tsm_out(c, st["loops"], st["err"], st["mean"])
    if kind == "contract":
        tsm.tsm_contract(ctx.h, c["prec"], st["seed"], 4, 3, st["s"], None, GAMMAS, st["moms"], st["out"])
        return _narrow(st["out"], c["prec"])
    tsm.tsm_net_forward(st["net"].h, ctx.h, 1, st["x"], st["y"])
    return torch.view_as_real(st["y"]).to(torch.bfloat16)   # BF16 operands on the tensor cores


def _tsm_out(c, loops, err, mean):
    per_site = 1.0 / (c["lx"] * c["ly"] * c["lz"])
    return {"loops": _narrow(loops * per_site, c["prec"]), "err": _narrow(err * per_site, c["prec"]),
            "lp_mean": _narrow(mean * per_site, c["prec"])}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    lx, ly, lz, lt = _dims_of(case)
    v = lx * ly * lz * lt
    kind, spinor, canon_links = case["kind"], 192.0, 4 * 144.0
    tier_links = 4.0 * (18 if case.get("prec") == F64 else 12) * REAL_BYTES.get(case.get("prec"), 4)
    hop = 1320.0 + 96
    if kind == "dslash":
        hops = {"full": 1.0, "schur": 1.0, "normal": 2.0}[case["op"]]   # in full-lattice applications
        half = 1.0 if case["op"] == "full" else 0.5                     # Schur fields live on the even sites
        return {"bytes": v * (spinor * half + spinor + tier_links), "flops": v * hops * hop}
    if kind == "gauge":
        return {"bytes": v * (canon_links + 2 * spinor + 4 * (18 * 8 + 12 * (4 + 2 + 2))), "flops": v * (hop + 4 * 250)}
    if kind == "solve":
        its = case["iters"] or 95   # what 1e-12 takes on these fields
        return {"bytes": v * (case["nrhs"] * 2 * spinor + tier_links),
                "flops": case["nrhs"] * v * ((2 * its + 2) * hop + its * 120)}
    if kind == "tsm":
        n = case["n_hp"] + case["n_lp"]
        outs = 16 * (lx * ly * lz if case["fft"] else case["nq"] * (1 + bin(case["deriv"]).count("1"))) * lt
        solve = n * (2 * case["iters"] + 2) + case["n_hp"] * 160
        con = 16 * 8.0 * case["nq"] * (1 + bin(case["deriv"]).count("1"))
        if case["fft"]:
            con = 16 * 5.0 * math.log2(lx * ly * lz)
        return {"bytes": v * (tier_links + 4 * 12 * 4) + outs * 40.0, "flops": v * (solve * hop + n * (con + 400))}
    if kind == "contract":
        return {"bytes": v * spinor + 16.0 * case["nq"] * lt * 16, "flops": v * (16 * 8.0 * case["nq"] + 400)}
    ch = _channels(case)
    mix = sum(8.0 * (4 * co) * (36 * ci) * 3 for ci, co in zip(ch[:-1], ch[1:]))
    return {"bytes": v * (2 * spinor + 4 * 48), "flops": v * (mix + 8 * 4 * 66 * sum(ch[:-1]))}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _gamma():
    s = torch.zeros(3, 2, 2, dtype=torch.complex128, device="cuda")
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    g = torch.zeros(4, 4, 4, dtype=torch.complex128, device="cuda")
    for k in range(3):
        g[k, :2, 2:], g[k, 2:, :2] = -1j * s[k], 1j * s[k]
    for a in range(2):
        g[3, a, 2 + a] = g[3, 2 + a, a] = 1
    return g, g[0] @ g[1] @ g[2] @ g[3]


def _insertions():
    g, g5 = _gamma()
    out = [torch.eye(4, dtype=torch.complex128, device="cuda")] + list(g) + [g5] + [m @ g5 for m in g]
    out += [0.5j * (g[m] @ g[n] - g[n] @ g[m]) for m, n in ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))]
    return torch.stack(out)


def _spin(m, psi):
    """m psi on the spin index (second to last); m has one or few entries per row."""
    rows = []
    for r in range(4):
        acc = 0
        for s in range(4):
            if m[r, s] != 0:
                acc = acc + m[r, s] * psi[..., s, :]
        rows.append(acc)
    return torch.stack(rows, dim=-2)


def _transport(U, psi, mu, forward):
    """U_mu(x) psi(x + mu) or U_mu(x - mu)^dagger psi(x - mu), antiperiodic in t."""
    ax, uax, lt = -3 - mu, 3 - mu, psi.shape[-6]
    q = torch.roll(psi, -1 if forward else 1, dims=ax)
    if mu == 3:
        sign = torch.ones(lt, dtype=torch.float64, device="cuda")
        sign[lt - 1 if forward else 0] = -1
        q = q * sign.reshape(lt, 1, 1, 1, 1, 1)
    u = U[..., mu, :, :] if forward else torch.roll(U[..., mu, :, :], 1, dims=uax).mH
    return (u[..., None, :, :] * q[..., None, :]).sum(-1)


class _Exact:
    def __init__(self, case, seed):
        self.U, self.dims = _links(_dims_of(case), seed), _dims_of(case)
        self.g, self.g5 = _gamma()
        lx, ly, lz, lt = self.dims
        ar = lambda n: torch.arange(n, device="cuda")
        par = (ar(lt)[:, None, None, None] + ar(lz)[:, None, None] + ar(ly)[:, None] + ar(lx)) % 2
        self.even = (par == 0).to(torch.float64)[..., None, None]
        self.sign5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device="cuda")[:, None]

    def hop(self, psi, dag=False):
        eye, s = torch.eye(4, dtype=torch.complex128, device="cuda"), -1.0 if dag else 1.0
        out = 0
        for mu in range(4):
            out = out + _spin(eye - s * self.g[mu], _transport(self.U, psi, mu, True))
            out = out + _spin(eye + s * self.g[mu], _transport(self.U, psi, mu, False))
        return out

    def twist(self, psi, mu, inverse=False):
        a = 1 + 2j * KAPPA * mu * self.sign5
        return psi / a if inverse else psi * a

    def full(self, psi):
        return self.twist(psi, MU) - KAPPA * self.hop(psi)

    def schur(self, e, dag=False):
        """Dhat e or Dhat^dag e on even-site fields (zero on the odd sites)."""
        if not dag:
            t = self.twist(self.hop(e) * (1 - self.even), MU, True)
            return e - KAPPA ** 2 * self.twist(self.hop(t) * self.even, MU, True)
        t = self.twist(self.hop(self.twist(e, -MU, True), True) * (1 - self.even), -MU, True)
        return e - KAPPA ** 2 * self.hop(t, True) * self.even

    def solve(self, b, tol, iters):
        """CG on the normal equations of the Schur complement from zero; b [n, ...]."""
        dot = lambda v: v.abs().square().flatten(1).sum(1)
        col = lambda v: v.reshape(-1, 1, 1, 1, 1, 1, 1)
        odd = 1 - self.even
        bh = self.twist(b * self.even + KAPPA * self.hop(self.twist(b * odd, MU, True)) * self.even, MU, True)
        r = self.schur(bh, True)
        x, p, rr = torch.zeros_like(r), r.clone(), dot(r)
        rr0 = rr.clone()
        for _ in range(iters):
            q = self.schur(p)
            alpha = rr / dot(q)
            x += col(alpha) * p
            r -= col(alpha) * self.schur(q, True)
            new = dot(r)
            if tol > 0 and bool((new < tol * tol * rr0).all()):
                break
            p = r + col(new / rr) * p
            rr = new
        return x + self.twist((b + KAPPA * self.hop(x)) * odd, MU, True)


def _philox_z4(dims, seed, source):
    """Z4 noise of one source: word 0 of Philox4x32-10 (Salmon et al., SC'11), two sign bits per component."""
    lx, ly, lz, lt = dims
    mask = 0xFFFFFFFF
    n = lx * ly * lz * lt
    c = [torch.arange(n, dtype=torch.int64, device="cuda")] + [torch.full((n,), v, dtype=torch.int64, device="cuda")
                                                                for v in (source, 0, 0)]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(a, m):
        lo, hi = a * (m & 0xFFFF), a * (m >> 16)
        return ((hi + (lo >> 16)) >> 16) & mask, (lo + ((hi & 0xFFFF) << 16)) & mask

    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    bits = (c[0][:, None] >> torch.arange(24, device="cuda")) & 1
    v = (1.0 - 2.0 * bits.to(torch.float64)).reshape(n, 12, 2) / math.sqrt(2.0)
    return torch.view_as_complex(v).reshape(lt, lz, ly, lx, 4, 3)


def _phases(dims, moms):
    lx, ly, lz, _ = dims
    ang = lambda n, L: 2 * math.pi * n / L * torch.arange(L, dtype=torch.float64, device="cuda")
    return torch.stack([torch.exp(1j * (ang(n[2], lz)[:, None, None] + ang(n[1], ly)[:, None] + ang(n[0], lx)))
                        for n in moms])


def _density(eta, s, ins):
    m = (eta.conj()[..., :, None, :] * s[..., None, :, :]).sum(-1)        # [T, Z, Y, X, 4, 4]
    return torch.stack([(m * g).sum((-2, -1)) for g in ins])             # [16, T, Z, Y, X]


def _project(dens, ph):
    return torch.einsum("qzyx,gtzyx->gqt", ph, dens)


def _exact_tsm(c, seed):
    ex, dims, ins = _Exact(c, seed), _dims_of(c), _insertions()
    ph = None if c["fft"] else _phases(dims, _momenta(c["nq"]))

    def value(eta, s):
        if c["fft"]:
            return torch.fft.ifftn(_density(eta, s, ins), dim=(2, 3, 4), norm="forward")
        out = [_project(_density(eta, s, ins), ph)]
        for mu in range(4):
            if c["deriv"] >> mu & 1:
                d = lambda f: _transport(ex.U, f, mu, True) - _transport(ex.U, f, mu, False)
                out.append(_project(0.25 * (_density(eta, d(s), ins) - _density(d(eta), s, ins)), ph))
        return torch.stack(out) if c["deriv"] else out[0]

    corr, lp, n_hp, n = [], [], c["n_hp"], c["n_hp"] + c["n_lp"]
    for j0 in range(0, n, 8):
        eta = torch.stack([_philox_z4(dims, seed, j) for j in range(j0, min(j0 + 8, n))])
        s = ex.solve(eta, 0.0, c["iters"])
        hp = min(n_hp - j0, len(eta))
        s_hp = ex.solve(eta[:hp], HP_TOL * 1e-2, 2000) if hp > 0 else None
        for k in range(len(eta)):
            v = value(eta[k], s[k])
            if k < hp:
                corr.append(value(eta[k], s_hp[k]) - v)
            else:
                lp.append(v)
    var, est = 0, 0
    for vals in (corr, lp):
        v = torch.stack(vals)
        est = est + v.mean(0)
        if len(vals) > 1:
            var = var + (v - v.mean(0)).abs().square().sum(0) / (len(vals) - 1) / len(vals)
    per_site = 1.0 / (dims[0] * dims[1] * dims[2])
    real = lambda x: torch.view_as_real((x * per_site).contiguous())
    return {"loops": real(est), "err": var.sqrt() * per_site, "lp_mean": real(torch.stack(lp).mean(0))}


def _momenta(nq):
    base = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    more = [(1, 1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, -1), (0, 1, 1), (0, -1, -1)]
    return {1: base[:1], 4: [base[0], base[1], base[3], base[5]], 7: base, 13: base + more}[nq]


def exact(case, seed):
    dims, kind = _dims_of(case), case["kind"]
    v = dims[0] * dims[1] * dims[2] * dims[3]
    if kind in ("dslash", "gauge"):
        ex, psi = _Exact(case, seed), _spinors(case, seed)
        op = case.get("op", "full")
        if op == "full":
            out = ex.full(psi)
        else:
            out = ex.schur(psi * ex.even)
            out = ex.schur(out, True) if op == "normal" else out
        return torch.view_as_real(out.contiguous()) if case["prec"] in (F16, BF16) else out
    if kind == "solve":
        ex, b = _Exact(case, seed), _z4(case, seed)
        if case["iters"]:
            return torch.view_as_real(torch.cat([ex.solve(x, 0.0, case["iters"]) for x in b.split(8)]))
        return ex.solve(b, 1e-15, 400)
    if kind == "tsm":
        if v * (case["n_hp"] + case["n_lp"]) * (1 + bin(case["deriv"]).count("1")) > 2.0e7:
            return None   # minutes in plain torch
        return _exact_tsm(case, seed)
    if kind == "contract":
        eta = _philox_z4(dims, seed, 3)
        return _project(_density(eta, _spinors(case, seed), _insertions()), _phases(dims, _momenta(case["nq"])))
    U, x = _links(dims, seed), _spinors(case, seed, 1)
    for w in _weights(case, seed):
        cin, cout = x.shape[0], w.shape[0] // 4
        w = w.reshape(cout * 4, 9, cin, 4)
        y = torch.zeros((cout * 4, v, 3), dtype=torch.complex128, device="cuda")
        for p in range(9):
            t = x if p == 0 else _transport(U, x, (p - 1) // 2, p % 2 == 1)
            y += torch.einsum("ocr,cvra->ova", w[:, p], t.reshape(cin, v, 4, 3))
        x = y.reshape(cout, 4, v, 3).transpose(1, 2).reshape((cout,) + tuple(reversed(dims)) + (4, 3))
    return torch.view_as_real(x[None].contiguous())
