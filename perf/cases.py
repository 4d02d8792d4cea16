"""The work that programs have this library do, as cases that can be timed.

A case is a dict of plain values; its "kind" says which public entry point it
calls:

  dw      one application of the Wilson-Dirac operator (psms_dw_apply)
  solve   one inversion of it, whole lattice or all Dirichlet blocks (psms_solve)
  logdet  the stochastic determinant-ratio estimates of one level of the
          filter (psms_logdet_ratio)
  sweep   the pure-gauge proposal (psms_gauge_sweep)
  lu      the exact block determinants (psms_block_logdet)
  filter  one whole step of the hierarchical filter (psms_filter_step)

Gauge fields are links U = exp(i eps H) to second order, reunitarised (eps =
0.5); where the operator is inverted they are thermalised at beta = 5.3 first,
as the method's are, and a second field is a domain proposal from the first
(both by the torch sweeps below with torch's random numbers, so that the inputs
do not hang on the library).
Quark fields and noise are Gaussian.  kappa = 0.156.

exact() computes the same outputs with plain torch in 64 bits on full-lattice
arrays [x0, x1, x2, x3, ...].
"""
import math

import torch

import paper_1204_1306_gb300 as ps

KAPPA = 0.156
A = 1.0 / (2.0 * KAPPA)
EPS = 0.5
BETA = 5.3
PRECS = {"f64": ps.PREC_F64, "f32": ps.PREC_F32, "bf16": ps.PREC_BF16}
DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
LEVELS = {"block": ps.LEVEL_BLOCK, "global": ps.LEVEL_GLOBAL, "sub": ps.LEVEL_SUB, "outer": ps.LEVEL_OUTER_GLOBAL}
MAXIT = 20000
THERM, THERM_OR = 3, 1  # thermalisation: iterations, overrelaxation sweeps


def listed():
    lat = "64x32x32x32"
    return [
        # the smallest lattice of the test suite: a call is a launch and its latency
        {"name": "dw f64 4^4", "kind": "dw", "dims": "4x4x4x4", "block": "2x2x2x2", "prec": "f64", "op": "full"},
        # the stand-alone operator on the largest lattice, each storage precision
        {"name": "dw f64 32^3x64", "kind": "dw", "dims": lat, "block": "4x4x4x4", "prec": "f64", "op": "full"},
        {"name": "dw f32 32^3x64", "kind": "dw", "dims": lat, "block": "4x4x4x4", "prec": "f32", "op": "full"},
        {"name": "dw bf16 32^3x64", "kind": "dw", "dims": lat, "block": "4x4x4x4", "prec": "bf16", "op": "full"},
        # one propagator on the ordinary lattice, mixed precision
        {"name": "solve 16^4", "kind": "solve", "dims": "16x16x16x16", "block": "4x4x4x4", "inner": "f32",
         "op": "full", "tol": 1e-12},
        # all blocks of one right-hand side on an odd number of blocks, fewer than the chip's SMs
        {"name": "solve blocks 12^4", "kind": "solve", "dims": "12x12x12x12", "block": "4x4x4x4", "inner": "f32",
         "op": "blocks", "tol": 1e-12},
        # the levels of the filter: block determinants, the global Schur complement, and the two
        # levels of the recursive decomposition with 8^4 domains of 4^4 blocks
        {"name": "block level 16^4", "kind": "logdet", "dims": "16x16x16x16", "block": "4x4x4x4", "level": "block",
         "n": 12, "inner": "f32", "tol": 1e-13, "outer": ""},
        {"name": "global level 16^4", "kind": "logdet", "dims": "16x16x16x16", "block": "4x4x4x4", "level": "global",
         "n": 12, "inner": "f32", "tol": 1e-13, "outer": ""},
        {"name": "domain level 16^4", "kind": "logdet", "dims": "16x16x16x16", "block": "4x4x4x4", "level": "sub",
         "n": 12, "inner": "f32", "tol": 1e-13, "outer": "8x8x8x8"},
        # the proposal of the largest lattice
        {"name": "sweep 32^3x64", "kind": "sweep", "dims": lat, "block": "4x4x4x4", "n_iter": 1, "n_or": 2},
        # exact determinants of sixteen 4^4 blocks (coefficient tuning on small lattices)
        {"name": "exact blocks 8^4", "kind": "lu", "dims": "8x8x8x8", "block": "4x4x4x4"},
        # the whole step on the ordinary lattice
        {"name": "filter step 16^4", "kind": "filter", "dims": "16x16x16x16", "block": "4x4x4x4", "n_block": 12,
         "n_global": 4, "n_or": 1, "inner": "f32", "tol": 1e-13},
    ]


def _lattice(rng, lo, hi, blocks, even_blocks=False, vb_max=4096):
    """Extents of a lattice of about a log-uniform volume in [lo, hi] and of its blocks."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        block = [rng.choice(blocks) for _ in range(4)]
        if rng.random() < 0.5:
            block = [block[0]] * 4
        dims = [b * rng.choice((2, 4, 6, 8, 12, 16) if even_blocks else (1, 2, 3, 4, 5, 6, 8, 12, 16)) for b in block]
        v, vb = math.prod(dims), math.prod(block)
        if vb <= vb_max and lo <= v <= hi and want / 1.6 <= v <= want * 1.6 and min(dims) >= 4 and max(dims) <= 64:
            return "x".join(map(str, dims)), "x".join(map(str, block))


def draw(rng):
    """Another case of the same ranges: even extents from 4 to 64, blocks of extents 2, 4 and 8."""
    kind = rng.choice(("dw", "dw", "solve", "solve", "logdet", "logdet", "sweep", "lu", "filter"))
    if kind == "dw":
        dims, block = _lattice(rng, 256, 1 << 21, (2, 4, 8))
        return {"kind": kind, "dims": dims, "block": block, "prec": rng.choice(("f64", "f32", "bf16")),
                "op": rng.choice(("full", "full", "blocks"))}
    if kind == "solve":
        dims, block = _lattice(rng, 256, 1 << 16, (2, 4, 8))
        op = rng.choice(("full", "blocks"))
        return {"kind": kind, "dims": dims, "block": block, "op": op, "tol": rng.choice((1e-10, 1e-12)),
                "inner": rng.choice(("f32", "f32", "f64"))}
    if kind == "logdet":
        level = rng.choice(("block", "block", "global"))
        dims, block = _lattice(rng, 256, 1 << 15, (2, 4), even_blocks=level == "global")
        return {"kind": kind, "dims": dims, "block": block, "level": level, "n": rng.randint(2, 16), "tol": 1e-13,
                "inner": rng.choice(("f32", "f32", "f64")), "outer": ""}
    if kind == "sweep":
        dims, block = _lattice(rng, 256, 1 << 21, (2, 4, 8))
        return {"kind": kind, "dims": dims, "block": block, "n_iter": 1, "n_or": rng.randint(0, 2)}
    if kind == "lu":
        dims, block = _lattice(rng, 256, 4096, (2, 4), vb_max=256)
        return {"kind": kind, "dims": dims, "block": block}
    dims, block = _lattice(rng, 256, 1 << 15, (2, 4), even_blocks=True)
    return {"kind": kind, "dims": dims, "block": block, "n_block": rng.randint(2, 12), "n_global": rng.randint(2, 6),
            "n_or": rng.randint(0, 2), "inner": "f32", "tol": 1e-13}


def _ints(s):
    return tuple(int(v) for v in s.split("x"))


# ---------------------------------------------------------------------------
# inputs, canonical arrays
# ---------------------------------------------------------------------------
def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 8 + what) & 0x7FFFFFFFFFFFFFFF)
    return g


def _reunit(u):
    """Gram-Schmidt on rows 0 and 1; row 2 = conj(row 0 x row 1).  u[..., 3, 3]."""
    r0, r1 = u[..., 0, :], u[..., 1, :]
    r0 = r0 / torch.sqrt((r0.abs() ** 2).sum(-1, keepdim=True))
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.sqrt((r1.abs() ** 2).sum(-1, keepdim=True))
    r2 = torch.stack([r0[..., 1] * r1[..., 2] - r0[..., 2] * r1[..., 1],
                      r0[..., 2] * r1[..., 0] - r0[..., 0] * r1[..., 2],
                      r0[..., 0] * r1[..., 1] - r0[..., 1] * r1[..., 0]], -1).conj()
    return torch.stack([r0, r1, r2], -2)


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _random_su3(n, eps, gen):
    """n SU(3) matrices: 1 + i eps H - eps^2 H^2 / 2 with Gaussian H, reunitarised."""
    out = torch.empty(n, 3, 3, dtype=torch.complex128, device="cuda")
    for lo in range(0, n, 1 << 20):
        m = min(1 << 20, n - lo)
        w = torch.randn(m, 8, dtype=torch.float64, device="cuda", generator=gen)
        h = torch.zeros(m, 3, 3, dtype=torch.complex128, device="cuda")
        is3 = 1.0 / math.sqrt(3.0)
        h[:, 0, 0] = w[:, 2] + is3 * w[:, 7]
        h[:, 1, 1] = -w[:, 2] + is3 * w[:, 7]
        h[:, 2, 2] = -2.0 * is3 * w[:, 7]
        for i, j, k in ((0, 1, 0), (0, 2, 3), (1, 2, 5)):
            z = torch.complex(w[:, k], -w[:, k + 1])
            h[:, i, j] = z
            h[:, j, i] = z.conj()
        x = 0.5j * eps * h
        out[lo:lo + m] = _reunit(torch.eye(3, device="cuda") + x + 0.5 * _mm(x, x))
    return out


def _coords(dims):
    return torch.meshgrid(*[torch.arange(L, device="cuda") for L in dims], indexing="ij")


def _active(dims, block):
    """bool [L0, L1, L2, L3, 4]: the links that a domain proposal changes (Sec. 3 of the paper; block None: all)."""
    if block is None:
        return torch.ones(dims + (4,), dtype=torch.bool, device="cuda")
    loc = [x % l for x, l in zip(_coords(dims), block)]
    act = torch.zeros(dims + (4,), dtype=torch.bool, device="cuda")
    small = min(block) <= 2

    def bnd(c):
        return ((c[0] == 0) | (c[0] == block[0] - 1) | (c[1] == 0) | (c[1] == block[1] - 1)
                | (c[2] == 0) | (c[2] == block[2] - 1) | (c[3] == 0) | (c[3] == block[3] - 1))

    b0 = bnd(loc)
    for mu in range(4):
        intra = loc[mu] != block[mu] - 1
        if small:
            act[..., mu] = intra
        else:
            c1 = [c + 1 if m == mu else c for m, c in enumerate(loc)]
            act[..., mu] = intra & ((b0.int() + bnd(c1).int()) <= 1)
    return act


def _field(dims, seed):
    n = math.prod(dims) * 4
    return _random_su3(n, EPS, _gen(seed, 0)).reshape(dims + (4, 3, 3))


def _spinor(dims, seed, dtype=torch.float64):
    """Gaussian quark field of unit variance per component, rounded to the storage type."""
    p = torch.randn(*dims, 4, 3, 2, dtype=torch.float64, device="cuda", generator=_gen(seed, 2)) * math.sqrt(0.5)
    return torch.view_as_complex(p.to(dtype).to(torch.float64))


def _flat(z):
    return torch.view_as_real(z.contiguous()).reshape(-1)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind, dims, block = case["kind"], _ints(case["dims"]), _ints(case["block"])
    n_fields = {"logdet": 2, "sweep": 2, "filter": 2}.get(kind, 1)
    ctx = ps.psms_create(dims, block, KAPPA, n_fields)
    ps.psms_set_stream(ctx, torch.cuda.current_stream())
    U = _thermal(dims, seed) if kind in ("solve", "logdet", "filter") else _field(dims, seed)
    ps.psms_gauge_set(ctx, 0, _flat(U))
    s = {"case": case, "ctx": ctx, "seed": seed}
    if kind in ("dw", "solve"):
        prec = case.get("prec", "f64")
        s["dtype"] = DTYPES[prec]
        s["in"] = torch.empty(ps.psms_spinor_bytes(ctx, PRECS[prec]), dtype=torch.uint8, device="cuda")
        s["out"] = torch.empty_like(s["in"])
        ps.psms_spinor_import(ctx, _flat(_spinor(dims, seed)), s["in"], PRECS[prec])
        s["op"] = ps.OP_FULL if case["op"] == "full" else ps.OP_BLOCKS
    elif kind == "logdet":
        ps.psms_gauge_set(ctx, 1, _flat(_proposal(U, block, seed)))
        if case["outer"]:
            ps.psms_set_outer_blocks(ctx, _ints(case["outer"]))
    elif kind in ("sweep", "filter"):
        s["links"] = torch.empty(U.numel() * 2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx, seed = s["case"], s["ctx"], s["seed"]
    kind = case["kind"]
    if kind == "dw":
        ps.psms_dw_apply(ctx, 0, s["op"], s["in"], s["out"], PRECS[case["prec"]])
        return s["out"].view(s["dtype"])
    if kind == "solve":
        ps.psms_solve(ctx, 0, s["op"], s["in"], s["out"], case["tol"], MAXIT, PRECS[case["inner"]])
        return s["out"].view(torch.float64)
    if kind == "logdet":
        return ps.psms_logdet_ratio(ctx, LEVELS[case["level"]], 0, 1, case["n"], ps.EST_INTERP, seed, 7, case["tol"],
                                    PRECS[case["inner"]])
    if kind == "lu":
        return ps.psms_block_logdet(ctx, 0)
    # slot 0 keeps the field before the call, as a chain does that may have to go back to it
    ps.psms_gauge_copy(ctx, 1, 0)
    if kind == "sweep":
        ps.psms_gauge_sweep(ctx, 1, ps.ACTIVE_BLOCKS, case["n_iter"], case["n_or"], BETA, seed, 0)
        ps.psms_gauge_get(ctx, 1, s["links"])
        return s["links"]
    r = ps.psms_filter_step(ctx, 1, beta0=BETA, n_iter=1, n_or=case["n_or"], n_block=case["n_block"],
                            n_global=case["n_global"], tol=case["tol"], inner_prec=PRECS[case["inner"]], seed=seed,
                            step=3)
    ps.psms_gauge_get(ctx, 1, s["links"])
    return {"links": s["links"], "delta_block": r["delta_block"], "delta_global": r["delta_global"],
            "accept_block": r["accept_block"], "accept_global": r["accept_global"]}


def work(case):
    """Bytes: links and fields in and out, once.  Flops: 1320 per site and application of the operator, times a
    nominal number of applications of the inversions (150 for a whole-lattice solve, 60 for the blocks)."""
    kind, dims, block = case["kind"], _ints(case["dims"]), _ints(case["block"])
    V = math.prod(dims)
    if kind == "dw":
        return {"bytes": {"f64": 960.0, "f32": 480.0, "bf16": 384.0}[case["prec"]] * V, "flops": 1320.0 * V}
    if kind == "solve":
        return {"bytes": (576.0 + 2 * 192.0) * V, "flops": 1320.0 * V * (150 if case["op"] == "full" else 60)}
    if kind == "sweep":
        if min(block) <= 2:
            links = sum((l - 1) / l for l in block)
        else:
            loc = math.prod(block)
            inner = [l - 2 for l in block]
            # links with at most one endpoint on the faces of the block
            links = sum((inner[m] + 1) * math.prod(inner[:m] + inner[m + 1:]) for m in range(4)) / loc
        # 3000 flop per update; each link field once in and once out
        return {"bytes": 2 * 576.0 * V, "flops": 3000.0 * links * V * case["n_iter"] * (2 + 2 * case["n_or"])}
    n = 6 * math.prod(block)
    if kind == "lu":
        return {"bytes": 576.0 * V, "flops": 8.0 / 3.0 * n ** 3 * V / math.prod(block)}
    apps = {"block": 61, "global": 122 + 150, "sub": 122 + 150, "outer": 122 + 450}
    if kind == "logdet":
        return {"bytes": 2 * 576.0 * V, "flops": 1320.0 * V * case["n"] * apps[case["level"]]}
    return {"bytes": 2 * 576.0 * V,
            "flops": 1320.0 * V * (case["n_block"] * apps["block"] + case["n_global"] * apps["global"])}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _e(mu, d, dag=False):
    """e_mu on the lower spin components d[..., 2, 3] (gamma_mu = [[0, e], [e^dagger, 0]]; e_0 = -1,
    e_k = -i sigma_k), or e_mu^dagger on the upper ones."""
    if mu == 0:
        return -d
    s = 1j if dag else -1j
    if mu == 1:
        return s * d.flip(-2)
    if mu == 2:
        q = torch.stack([-d[..., 1, :], d[..., 0, :]], -2)
        return -q if dag else q
    return torch.stack([s * d[..., 0, :], -s * d[..., 1, :]], -2)


class _Ops:
    """D of one gauge field U[L0, L1, L2, L3, 4, 3, 3]; mode full, block (hops inside the blocks) or inter."""

    def __init__(self, U, block, mode):
        dims = U.shape[:4]
        self.mode = mode
        loc = [x % l for x, l in zip(_coords(dims), block)]
        self.fwd, self.bwd = [], []
        for mu in range(4):
            u = U[..., mu, :, :]
            f = torch.ones(dims, dtype=torch.float64, device="cuda")
            if mu == 0:
                f[-1] = -1.0  # antiperiodic in time
            inside = (loc[mu] != block[mu] - 1).double()
            if mode == "block":
                f = f * inside
            if mode == "inter":
                f = f * (1.0 - inside)
            w = u * f[..., None, None]
            self.fwd.append(w.contiguous())
            self.bwd.append(torch.roll(w, 1, mu).conj().transpose(-1, -2).contiguous())

    def __call__(self, psi, dag=False):
        out = torch.zeros_like(psi) if self.mode == "inter" else A * psi
        up, dn = psi[..., :2, :], psi[..., 2:, :]
        s = -1.0 if dag else 1.0
        for mu in range(4):
            for w, t, sh in ((self.fwd[mu], -s, -1), (self.bwd[mu], s, 1)):
                h = torch.roll(up + t * _e(mu, dn), sh, mu)
                h = (w[..., None, :, :] * h[..., :, None, :]).sum(-1)
                out[..., :2, :] -= 0.5 * h
                out[..., 2:, :] -= (0.5 * t) * _e(mu, h, dag=True)
        return out


def _invert(D, b):
    """D^-1 b to about 1e-15: conjugate gradients on the normal equations, restarted from the true residual."""
    x = torch.zeros_like(b)
    bn = float((b.abs() ** 2).sum())
    if bn == 0.0:
        return x
    for _ in range(4):
        r = b - D(x)
        start = float((r.abs() ** 2).sum())
        if start <= 1e-30 * bn:
            break
        e, s = torch.zeros_like(b), D(r, dag=True)
        p, g, target = s, (s.abs() ** 2).sum(), max(1e-15 * start, 1e-31 * bn)
        for it in range(2000):
            q = D(p)
            al = g / (q.abs() ** 2).sum()
            e += al * p
            r -= al * q
            if it % 10 == 9 and float((r.abs() ** 2).sum()) <= target:
                break
            s = D(r, dag=True)
            g, old = (s.abs() ** 2).sum(), g
            p = s + (g / old) * p
        x += e
    return x


def _site_order(dims, block):
    """Position of every lattice site in a native field: parity, then the blocks (all even-colour ones first where
    the blocks form a checkerboard), then half the place within the block."""
    x = _coords(dims)
    nb = [L // l for L, l in zip(dims, block)]
    B = [c // l for c, l in zip(x, block)]
    b = ((B[0] * nb[1] + B[1]) * nb[2] + B[2]) * nb[3] + B[3]
    if all(n % 2 == 0 for n in nb):
        b = ((B[0] + B[1] + B[2] + B[3]) % 2) * (math.prod(nb) // 2) + b // 2
    y = [c % l for c, l in zip(x, block)]
    loc = ((y[0] * block[1] + y[1]) * block[2] + y[2]) * block[3] + y[3]
    p = (x[0] + x[1] + x[2] + x[3]) % 2
    return (p * (math.prod(dims) // 2) + b * (math.prod(block) // 2) + loc // 2).reshape(-1)


def _native(psi, dims, block, per):
    """psi in the native order: units of `per` complex components, site fastest."""
    V = math.prod(dims)
    out = torch.empty(V, 12, dtype=torch.complex128, device="cuda")
    out[_site_order(dims, block)] = psi.reshape(V, 12)
    return _flat(out.reshape(V, 12 // per, per).transpose(0, 1))


def _s64(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _mulhilo(m, b):
    """(high, low) 64 bits of m * b, b an int64 tensor of unsigned words."""
    M = 0xFFFFFFFF
    a0, a1, b0, b1 = m & M, m >> 32, b & M, (b >> 32) & M
    p00, p01, p10, p11 = a0 * b0, a0 * b1, a1 * b0, a1 * b1
    mid = ((p00 >> 32) & M) + (p01 & M) + (p10 & M)
    return p11 + ((p01 >> 32) & M) + ((p10 >> 32) & M) + ((mid >> 32) & M), _s64(m) * b


def _uniforms(seed, tag, *ctr):
    """Philox-4x64-10 of the counters, as four uniforms each (Salmon et al., SC'11)."""
    c = torch.broadcast_tensors(*[torch.as_tensor(v, dtype=torch.int64, device="cuda") for v in ctr])
    c0, c1, c2, c3 = (v.clone() for v in c)
    for r in range(10):
        k0, k1 = ((seed + r * 0x9E3779B97F4A7C15) % (1 << 64), (tag + r * 0xBB67AE8584CAA73B) % (1 << 64))
        h0, l0 = _mulhilo(0xD2E7470EE14C6C93, c0)
        h1, l1 = _mulhilo(0xCA5A826395121157, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ _s64(k0), l1, h0 ^ c3 ^ _s64(k1), l0
    return [(((w >> 12) & ((1 << 52) - 1)).double() + 0.5) * 2.0 ** -52 for w in (c0, c1, c2, c3)]


def _noise(dims, seed, counter, level, i):
    site = torch.arange(math.prod(dims), device="cuda")
    z = []
    for j in range(6):
        u = _uniforms(seed, 2, counter, (level << 32) | i, site, j)
        for m in range(2):
            z.append(torch.polar(torch.sqrt(-torch.log(u[2 * m])), 2.0 * math.pi * u[2 * m + 1]))
    return torch.stack(z, -1).reshape(dims + (4, 3))


def _projector(dims, block):
    """(sites on two or more faces, [(mu, sign, sites on this face alone)]) of the even-colour blocks."""
    x = _coords(dims)
    loc = [c % l for c, l in zip(x, block)]
    black = sum(c // l for c, l in zip(x, block)) % 2 == 0
    faces = [(mu, sg, loc[mu] == (block[mu] - 1 if sg > 0 else 0)) for mu in range(4) for sg in (1.0, -1.0)]
    n = sum(f.int() for _, _, f in faces)
    return black & (n >= 2), [(mu, sg, f & black & (n == 1)) for mu, sg, f in faces]


def _project(P, v):
    out = v * P[0][..., None, None]
    for mu, t, f in P[1]:
        h = 0.5 * (v[..., :2, :] + t * _e(mu, v[..., 2:, :])) * f[..., None, None]
        out[..., :2, :] += h
        out[..., 2:, :] += t * _e(mu, h, dag=True)
    return out


def _exact_levels(case, seed, dims, block):
    n = case["n"]
    U = _thermal(dims, seed)
    Up = _proposal(U, block, seed)
    nb = [L // l for L, l in zip(dims, block)]
    black = (sum(c // l for c, l in zip(_coords(dims), block)) % 2 == 0)[..., None, None]
    got = []
    for i in range(n):
        Ua, Ub = ((n - i) / n) * U + (i / n) * Up, ((n - i - 1) / n) * U + ((i + 1) / n) * Up
        if case["level"] == "block":
            xi = _noise(dims, seed, 7, 1, i)
            y = _invert(_Ops(Ub, block, "block"), _Ops(Ua, block, "block")(xi))
            d = (y.abs() ** 2 - xi.abs() ** 2).sum((-1, -2))
            d = d.reshape(nb[0], block[0], nb[1], block[1], nb[2], block[2], nb[3], block[3])
            got.append(d.sum((1, 3, 5, 7)).reshape(-1))
        else:
            P = _projector(dims, block)
            xi = _project(P, _noise(dims, seed, 7, 2, i))
            inter, blocks = _Ops(Ua, block, "inter"), _Ops(Ua, block, "block")
            t = _invert(blocks, inter(xi) * ~black)
            v = xi - _project(P, _invert(blocks, inter(t) * black))
            w = v - _project(P, _invert(_Ops(Ub, block, "full"), _Ops(Ub, block, "inter")(v) * ~black))
            got.append((w.abs() ** 2 - xi.abs() ** 2).sum().reshape(1))
    return torch.stack(got, 1) if case["level"] == "block" else torch.cat(got)


def _swept(U0, block, n_iter, n_or, draws):
    """The proposal on the active links (block None: on all): Cabibbo-Marinari heatbath (Kennedy-Pendleton, Creutz)
    and overrelaxation over the checkerboard subsets, in both orders; U0[L0, L1, L2, L3, 4, 3, 3].
    draws(sweep, links, code, attempt): four uniforms per link."""
    dims = tuple(U0.shape[:4])
    V = math.prod(dims)
    U = U0.reshape(V, 4, 3, 3).clone()
    x = [c.reshape(-1) for c in _coords(dims)]
    act = _active(dims, block).reshape(V, 4)
    parity = sum(x) % 2
    cols = (None,)
    if block is not None and min(block) <= 2:
        cols, colour = (0, 1), sum(c // l for c, l in zip(x, block)) % 2
    subs = [(mu, torch.nonzero(act[:, mu] & (parity == p) & ((colour == c) if c is not None else True)).reshape(-1))
            for c in cols for mu in range(4) for p in (0, 1)]
    strides = (dims[1] * dims[2] * dims[3], dims[2] * dims[3], dims[3], 1)

    def shift(s, mu, d):
        c = (s // strides[mu]) % dims[mu]
        return s + (((c + d) % dims[mu]) - c) * strides[mu]

    def dagger(m):
        return m.conj().transpose(-1, -2)

    def quat(q):
        q = [torch.as_tensor(v) for v in q]
        return torch.stack([torch.complex(q[0], q[3]), torch.complex(q[2], q[1]), torch.complex(-q[2], q[1]),
                            torch.complex(q[0], -q[3])], -1).reshape(-1, 2, 2)

    def a0_draw(al, link, sweep, code):
        a0, left = torch.ones_like(al), torch.arange(al.numel(), device="cuda")
        for attempt in range(1000):
            if not left.numel():
                break
            u, a = draws(sweep, link[left], code, attempt), al[left]
            xx = -(torch.log(u[0]) + torch.cos(2.0 * math.pi * u[1]) ** 2 * torch.log(u[2])) / a
            cr = 1.0 + torch.log(u[0] + (1.0 - u[0]) * torch.exp(-2.0 * a)) / a
            kp = a >= 2.0
            ok = torch.where(kp, u[3] ** 2 <= 1.0 - 0.5 * xx, u[1] ** 2 <= 1.0 - cr * cr)
            a0[left[ok]] = torch.where(kp, 1.0 - xx, cr)[ok]
            left = left[~ok]
        return a0

    def update(mu, s, heat, sweep):
        A_ = torch.zeros(s.numel(), 3, 3, dtype=torch.complex128, device="cuda")
        for nu in range(4):
            if nu != mu:
                m = shift(s, nu, -1)
                A_ += _mm(_mm(U[shift(s, mu, 1), nu], dagger(U[shift(s, nu, 1), mu])), dagger(U[s, nu]))
                A_ += _mm(_mm(dagger(U[shift(m, mu, 1), nu]), dagger(U[m, mu])), U[m, nu])
        Ul, link = U[s, mu].clone(), 4 * s + mu
        forward = draws(sweep, link, 0, 0)[0] < 0.5
        at = torch.arange(s.numel(), device="cuda")
        for k in range(3):
            sg = torch.where(forward, k, 2 - k)
            i, j = torch.where(sg == 2, 1, 0), torch.where(sg == 0, 1, 2)
            W = _mm(Ul, A_)
            w = [W[at, i, i], W[at, i, j], W[at, j, i], W[at, j, j]]
            r = [0.5 * (w[0] + w[3]).real, 0.5 * (w[1] + w[2]).imag, 0.5 * (w[1] - w[2]).real, 0.5 * (w[0] - w[3]).imag]
            kn = torch.sqrt(sum(v * v for v in r))
            vd = quat([r[0] / kn, -r[1] / kn, -r[2] / kn, -r[3] / kn])
            if heat:
                a0 = a0_draw(2.0 * BETA * kn / 3.0, link, sweep, 1 + 2 * k)
                u = draws(sweep, link, 2 + 2 * k, 0)
                cth, phi = 2.0 * u[0] - 1.0, 2.0 * math.pi * u[1]
                sth, rad = torch.sqrt((1.0 - cth * cth).clamp(min=0.0)), torch.sqrt((1.0 - a0 * a0).clamp(min=0.0))
                vd = _mm(quat([a0, rad * sth * torch.cos(phi), rad * sth * torch.sin(phi), rad * cth]), vd)
            else:
                vd = _mm(vd, vd)
            ri, rj = Ul[at, i], Ul[at, j]
            Ul[at, i] = vd[:, 0, 0, None] * ri + vd[:, 0, 1, None] * rj
            Ul[at, j] = vd[:, 1, 0, None] * ri + vd[:, 1, 1, None] * rj
        U[s, mu] = Ul

    sweep = 0
    for _ in range(n_iter):
        for heat, rev in [(True, False)] + [(False, False)] * n_or + [(False, True)] * n_or + [(True, True)]:
            for mu, s in (subs[::-1] if rev else subs):
                if s.numel():
                    update(mu, s, heat, sweep)
            sweep += 1
    U[act] = _reunit(U[act])
    return U.reshape(U0.shape)


def _torch_draws(gen):
    def draws(sweep, link, code, attempt):
        u = torch.rand(4, link.numel(), dtype=torch.float64, device="cuda", generator=gen)
        return u.clamp(2.0 ** -53, 1.0 - 2.0 ** -53)
    return draws


def _thermal(dims, seed):
    return _swept(_field(dims, seed), None, THERM, THERM_OR, _torch_draws(_gen(seed, 3)))


def _proposal(U, block, seed):
    return _swept(U, block, 1, 1, _torch_draws(_gen(seed, 1)))


def _exact_lu(seed, dims, block):
    """ln |det D_b| of the dense block operators on the odd sites: A^{n_e} det(A - D_oe D_eo / A)."""
    U = _field(dims, seed)
    vb = math.prod(block)
    par = (sum(_coords(block)) % 2).reshape(-1)
    got = []
    for b0 in range(0, dims[0], block[0]):
        for b1 in range(0, dims[1], block[1]):
            for b2 in range(0, dims[2], block[2]):
                for b3 in range(0, dims[3], block[3]):
                    u = U[b0:b0 + block[0], b1:b1 + block[1], b2:b2 + block[2], b3:b3 + block[3]]
                    D = torch.zeros(vb, 4, 3, vb, 4, 3, dtype=torch.complex128, device="cuda")
                    g = torch.arange(vb, device="cuda").reshape(block)
                    for mu in range(4):
                        x, y = g.narrow(mu, 0, block[mu] - 1).reshape(-1), g.narrow(mu, 1, block[mu] - 1).reshape(-1)
                        w = u[..., mu, :, :].reshape(vb, 3, 3)[x]
                        e = _e(mu, torch.eye(2, dtype=torch.complex128, device="cuda").reshape(2, 2)[:, :, None])[..., 0]
                        e = e.T  # e[s, t]
                        one = torch.eye(2, dtype=torch.complex128, device="cuda")
                        for t, src, dst, m in ((-1.0, y, x, w), (1.0, x, y, w.conj().transpose(-1, -2))):
                            spin = torch.cat([torch.cat([one, t * e], 1), torch.cat([t * e.conj().T, one], 1)], 0)
                            blk = -0.5 * spin[None, :, None, :, None] * m[:, None, :, None, :]
                            D[dst, :, :, src, :, :] += blk
                    D = D.reshape(vb, 12, vb, 12)
                    o, ev = torch.nonzero(par == 1).reshape(-1), torch.nonzero(par == 0).reshape(-1)
                    oe = D[o][:, :, ev].reshape(6 * vb, 6 * vb)
                    eo = D[ev][:, :, o].reshape(6 * vb, 6 * vb)
                    M = A * torch.eye(6 * vb, dtype=torch.complex128, device="cuda") - (oe @ eo) / A
                    got.append(6 * vb * math.log(A) + torch.linalg.slogdet(M).logabsdet)
    return torch.stack(got)


def exact(case, seed):
    kind, dims, block = case["kind"], _ints(case["dims"]), _ints(case["block"])
    if kind in ("dw", "solve"):
        U = _field(dims, seed) if kind == "dw" else _thermal(dims, seed)
        D = _Ops(U, block, "full" if case["op"] == "full" else "block")
        if kind == "dw":
            per = {"f64": 1, "f32": 2, "bf16": 4}[case["prec"]]
            return _native(D(_spinor(dims, seed, DTYPES[case["prec"]])), dims, block, per)
        return _native(_invert(D, _spinor(dims, seed)), dims, block, 1)
    if kind == "logdet" and case["level"] in ("block", "global"):
        # about 1 s (block) and 4 s (global) a noise vector at 16^4
        if math.prod(dims) * case["n"] * (1 if case["level"] == "block" else 4) > 16 * 16 ** 4:
            return None
        return _exact_levels(case, seed, dims, block)
    if kind == "sweep":
        def draws(sweep, link, code, attempt):
            return _uniforms(seed, 3, sweep, link, code, attempt)
        return _flat(_swept(_field(dims, seed), block, case["n_iter"], case["n_or"], draws))
    if kind == "lu":
        return _exact_lu(seed, dims, block)
    return None  # the whole step and the recursive levels are minutes of the work above
