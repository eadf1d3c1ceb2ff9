"""The work this library does for its users, as timed cases.

Every case goes through the public entry points of ``paper_1111_0125_gb300``
with the inputs a lattice program has in hand: a gauge handle made once per
configuration (SU(3) links exp(i eps H), projected, phases not folded), Gaussian
fields already in the device layout for the operators, canonical Gaussian
sources for the solvers.

Operators (``op``):
  dslash      one half-pass D_{p <- 1-p}                  (stg_dslash)
  a_dot       A = m^2 - D_eo D_oe with d^dag A d           (stg_apply_A_dot)
  group       half-passes on several small lattices at once (stg_dslash_group)
  a_mrhs      A on several fields of one lattice           (stg_apply_A_mrhs)
  solve       one CG solve                                 (stg_cg_solve)
  solve_mrhs  one batched CG solve                         (stg_cg_solve_mrhs)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1111_0125_gb300 as stg

PREC = {"f64": stg.STG_FP64, "f32": stg.STG_FP32, "f16": stg.STG_FP16, "fx16": stg.STG_FX16,
        "bf16": stg.STG_BF16}
LINK_BYTES = {("f64", 18): 144, ("f64", 12): 96, ("f32", 18): 72, ("f32", 12): 48}
FIELD_BYTES = {"f64": 48, "f32": 24}


def _case(name, op, prec, recon, dims, **more):
    c = {"name": name, "op": op, "prec": prec, "recon": recon,
         "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3]}
    c.update(more)
    return c


def listed():
    return [
        # one operator application on the smallest served lattice: latency and launch
        _case("dslash_f32_8x8x8x8", "dslash", "f32", 12, (8, 8, 8, 8)),
        # the serving layer's small lattices in one launch: 8^4 and 12^3x24 in turn
        _case("group_f32_8_lattices", "group", "f32", 12, (12, 12, 12, 24), n=8),
        # a user's own CG or eigensolver in single precision on an ordinary lattice
        _case("a_dot_f32_16x16x16x32", "a_dot", "f32", 12, (16, 16, 16, 32), mass=0.01),
        # the double-precision operator: plain CG and every true residual
        _case("a_dot_f64_24x24x24x48", "a_dot", "f64", 18, (24, 24, 24, 48), mass=0.01),
        # the largest lattice, 16-bit storage: the bandwidth-bound inner operator
        _case("a_dot_f16_32x32x32x64", "a_dot", "f16", 12, (32, 32, 32, 64), mass=0.005),
        # bfloat16 storage with uncompressed links on extents that fill no block evenly
        _case("dslash_bf16_20x14x18x22", "dslash", "bf16", 18, (20, 14, 18, 22)),
        # 16 right-hand sides on one gauge field (propagators of one configuration)
        _case("a_mrhs_f32_24x24x24x48_n16", "a_mrhs", "f32", 12, (24, 24, 24, 48), n=16, mass=0.005),
        # a few right-hand sides (not a multiple of the register block) on a served lattice
        _case("a_mrhs_f32_12x12x12x24_n5", "a_mrhs", "f32", 12, (12, 12, 12, 24), n=5, mass=0.005),
        # complete mixed-precision solves: the smallest served lattice ...
        _case("solve_f32_8x8x8x8", "solve", "f32", 12, (8, 8, 8, 8), mass=0.05, eps=0.5),
        # ... the ordinary one with FP32 inner iterations ...
        _case("solve_f32_16x16x16x32", "solve", "f32", 12, (16, 16, 16, 32), mass=0.01, eps=0.4),
        # ... and a large one with 16-bit inner iterations (the inner solver for big lattices)
        _case("solve_f16_24x24x24x48", "solve", "f16", 12, (24, 24, 24, 48), mass=0.01, eps=0.5),
        # a batch of systems with their own masses on one served field
        _case("solve_mrhs_f32_12x12x12x24_n8", "solve_mrhs", "f32", 12, (12, 12, 12, 24), n=8,
              mass=0.01, eps=0.5),
    ]


def _dims_near(rng, volume):
    """Even extents with a volume near the one asked for: Lt up to 64, space up to 32."""
    while True:
        lt = 2 * rng.randint(2, 32)
        space = [2 * rng.randint(2, 16) for _ in range(3)]
        v = lt * space[0] * space[1] * space[2]
        if 0.7 * volume <= v <= min(1.4 * volume, 2097152):
            return (*space, lt)


def draw(rng):
    op = rng.choice(["dslash", "dslash", "a_dot", "a_dot", "group", "a_mrhs", "solve", "solve_mrhs"])
    top = {"dslash": 2097152, "a_dot": 2097152, "group": 41472, "a_mrhs": 663552, "solve": 200000,
           "solve_mrhs": 50000}[op]
    dims = _dims_near(rng, math.exp(rng.uniform(math.log(4096), math.log(top))))
    volume = dims[0] * dims[1] * dims[2] * dims[3]
    c = _case("", op, "f32", 12, dims)
    del c["name"]
    if op == "dslash":
        c["prec"] = rng.choice(["f64", "f32", "f16", "bf16"])
        c["recon"] = rng.choice([12, 12, 18])
    elif op == "a_dot":
        c["prec"] = rng.choice(["f64", "f64", "f32", "f16"])
        c["recon"] = rng.choice([12, 18])
        c["mass"] = round(math.exp(rng.uniform(math.log(0.005), math.log(0.1))), 5)
    elif op == "group":
        c["recon"] = rng.choice([12, 18])
        c["n"] = rng.randint(2, 16)
    elif op == "a_mrhs":
        c["n"] = rng.randint(2, max(2, min(16, 16 * 663552 // volume)))
        c["mass"] = 0.005
    else:
        c["mass"] = round(math.exp(rng.uniform(math.log(0.005), math.log(0.1))), 5)
        c["eps"] = rng.choice([0.4, 0.5, 0.6])
        if op == "solve":
            c["prec"] = rng.choice(["f64", "f32", "f32", "f16", "fx16"])
        else:
            c["prec"] = rng.choice(["f32", "f32", "fx16"])
            c["n"] = rng.randint(2, 8)
    return c


# ---------------------------------------------------------------------------
# inputs, made on the GPU from the seed
# ---------------------------------------------------------------------------
def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _group_dims(case):
    """The lattices of a group: 8^4 and the case's own extents in turn."""
    return [_dims(case) if k % 2 else (8, 8, 8, 8) for k in range(case["n"])]


def _gaussian(gen, shape):
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device="cuda",
                                             generator=gen)) * math.sqrt(0.5)


def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _links(gen, dims, eps):
    """SU(3) links near exp(i eps H), H Gaussian traceless Hermitian: a Taylor
    sum, then rows 0 and 1 made orthonormal and row 2 = conj(row 0 x row 1)."""
    lx, ly, lz, lt = dims
    n = lx * ly * lz * lt * 4
    u = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    for s in range(0, n, 1 << 21):
        m = min(1 << 21, n - s)
        g = _gaussian(gen, (m, 3, 3))
        h = 0.5 * (g + g.mH)
        h = h - h.diagonal(dim1=-2, dim2=-1).sum(-1)[:, None, None] / 3 * eye
        h = h * (1j * eps)
        e = eye + h / 4
        for k in (3, 2, 1):
            e = eye + _mm(h, e) / k
        r0 = e[:, 0] / torch.linalg.vector_norm(e[:, 0], dim=-1, keepdim=True)
        r1 = e[:, 1] - (r0.conj() * e[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        u[s:s + m] = torch.stack([r0, r1, torch.linalg.cross(r0, r1, dim=-1).conj()], dim=1)
    return u.view(lt, lz, ly, lx, 4, 3, 3)


def _masses(case):
    """The batch's masses, log-spaced from the case's mass to ten times that."""
    n = case["n"]
    return [case["mass"] * 10.0 ** (k / max(1, n - 1)) for k in range(n)]


def _drawn(case, seed):
    """[(dims, links, canonical fields (k, Vh, 3))] of the case's lattices."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    out = []
    for dims in (_group_dims(case) if case["op"] == "group" else [_dims(case)]):
        u = _links(gen, dims, case.get("eps", 0.5))
        vh = dims[0] * dims[1] * dims[2] * dims[3] // 2
        k = case["n"] if case["op"] in ("a_mrhs", "solve_mrhs") else 1
        out.append((dims, u, _gaussian(gen, (k, vh, 3))))
    return out


def prepare(case, seed):
    op, prec = case["op"], PREC[case["prec"]]
    st = {"op": op, "prec": prec, "mass": case.get("mass", 0.0), "tol": 1e-10, "gauges": [],
          "ins": [], "outs": [], "values": []}
    for dims, u, chi in _drawn(case, seed):
        g = stg.Gauge(dims, u.cpu().numpy(), sloppy=prec, recon=case["recon"])
        st["gauges"].append(g)
        if op in ("solve", "solve_mrhs"):
            st["ins"].append(chi)
            continue
        st["ins"].append(torch.cat([g.pack(c, prec) for c in chi]))
        st["outs"].append(torch.empty_like(st["ins"][-1]))
        st["values"].append(_values(st["outs"][-1], case["prec"]))
    if op in ("a_mrhs", "solve_mrhs"):
        st["masses"] = np.asarray(_masses(case))
    if op == "a_dot":
        st["dot"] = torch.empty(1, dtype=torch.float64, device="cuda")
    if op == "group":
        st["handles"] = [g.handle for g in st["gauges"]]
    torch.cuda.synchronize()
    return st


def _values(field, kind):
    """A device-layout field as its numbers: one tensor, or the 16-bit values and scales."""
    if kind == "f64":
        return field.view(torch.float64)
    if kind == "f32":
        return field.view(torch.float32)
    half = torch.float16 if kind == "f16" else torch.bfloat16
    return [field.view(half).view(-1, 8)[:, :6], field.view(torch.float32).view(-1, 4)[:, 3]]


def run(state):
    op, prec, g = state["op"], state["prec"], state["gauges"][0]
    if op == "dslash":
        stg.stg_dslash(g.handle, 0, state["ins"][0], state["outs"][0], prec)
        return state["values"]
    if op == "a_dot":
        stg.stg_apply_A_dot(g.handle, state["mass"], state["ins"][0], state["outs"][0], state["dot"], prec)
        return [state["values"][0], state["dot"]]
    if op == "group":
        stg.stg_dslash_group(state["handles"], [0] * len(state["handles"]), state["ins"], state["outs"], prec)
        return state["values"]
    if op == "a_mrhs":
        stg.stg_apply_A_mrhs(g.handle, len(state["masses"]), state["masses"], state["ins"][0],
                             state["outs"][0], prec)
        return state["values"]
    b = state["ins"][0]
    x = torch.zeros_like(b)
    if op == "solve":
        stg.stg_cg_solve(g.handle, b, x, state["mass"], state["tol"])
    else:
        stg.stg_cg_solve_mrhs(g.handle, len(state["masses"]), b, x, state["masses"], state["tol"])
    return x


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _iterations(case):
    """CG iterations to 1e-10 on these random links, to a factor of about 1.5:
    they follow the smallest eigenvalue of D, which falls with the volume and
    with the roughness of the links (measured, eps 0.5: 217 on 8^4, 556 on
    12^3x24, 862 on 24^3x48; eps 0.4: 351 on 16^3x32)."""
    v = case["lx"] * case["ly"] * case["lz"] * case["lt"]
    return 215.0 * (v / 4096.0) ** 0.27 * (2.0 * case["eps"]) ** 2


def work(case):
    """Each input read once and each output written once; links of a
    compressed handle by their compressed size; the solves as so many
    iterations of two half-passes, d, q, t, y and r once each."""
    op, prec = case["op"], case["prec"]
    link = LINK_BYTES.get((prec, case["recon"]), 24 if case["recon"] == 12 else 36)
    field = FIELD_BYTES.get(prec, 16)
    vh = case["lx"] * case["ly"] * case["lz"] * case["lt"] // 2
    n = case.get("n", 1)
    if op == "dslash":
        return {"bytes": vh * (8 * link + 2 * field), "flops": 576 * vh}
    if op == "a_dot":
        return {"bytes": vh * (8 * link + 2 * field) + 8, "flops": (2 * 576 + 24) * vh}
    if op == "group":
        sites = sum(d[0] * d[1] * d[2] * d[3] // 2 for d in _group_dims(case))
        return {"bytes": sites * (8 * link + 2 * field), "flops": 576 * sites}
    if op == "a_mrhs":
        return {"bytes": vh * (8 * link + 2 * n * field), "flops": n * (2 * 576 + 12) * vh}
    wide = 48 if prec == "f64" else 24
    it = _iterations(case)
    per_site = 8 * link + n * (3 * field + 2 * wide)
    return {"bytes": it * vh * per_site, "flops": it * n * (2 * 576 + 60) * vh}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
class _Plain:
    """D and A on checkerboard fields (Vh, 3) by index tables."""

    def __init__(self, dims, u):
        lx, ly, lz, lt = dims
        dev = u.device
        lex = torch.arange(lx * ly * lz * lt, device=dev)
        x = [lex % lx, lex // lx % ly, lex // (lx * ly) % lz, lex // (lx * ly * lz)]
        parity = (x[0] + x[1] + x[2] + x[3]) % 2
        step = [1, lx, lx * ly, lx * ly * lz]
        u = u.reshape(-1, 4, 3, 3)
        self.hops = {}
        for p in (0, 1):
            at = lex[parity == p]
            for mu in range(4):
                c = x[mu][at]
                fwd = at + torch.where(c == dims[mu] - 1, -(dims[mu] - 1) * step[mu], step[mu])
                bwd = at + torch.where(c == 0, (dims[mu] - 1) * step[mu], -step[mu])
                eta = 1.0 - 2.0 * (sum([x[nu][at] for nu in range(mu)], torch.zeros_like(at)) % 2)
                sf = eta * (torch.where(c == lt - 1, -1.0, 1.0) if mu == 3 else 1.0)
                sb = eta * (torch.where(c == 0, -1.0, 1.0) if mu == 3 else 1.0)
                self.hops[p, mu, 0] = (u[at, mu] * sf[:, None, None], fwd >> 1)
                self.hops[p, mu, 1] = ((u[bwd, mu] * -sb[:, None, None]).mH.contiguous(), bwd >> 1)

    def dslash(self, p, chi):
        out = torch.zeros_like(chi)
        for mu in range(4):
            for way in (0, 1):
                m, j = self.hops[p, mu, way]
                out += (m * chi[j].unsqueeze(-2)).sum(-1)
        return out

    def a(self, mass, chi):
        return mass * mass * chi - self.dslash(0, self.dslash(1, chi))

    def solve(self, mass, b):
        x = torch.zeros_like(b)
        r = b.clone()
        d, rr = r.clone(), torch.linalg.vector_norm(r) ** 2
        stop = (1e-14 * float(torch.linalg.vector_norm(b))) ** 2
        for k in range(20000):
            q = self.a(mass, d)
            alpha = rr / (d.conj() * q).sum().real
            x += alpha * d
            r -= alpha * q
            new = torch.linalg.vector_norm(r) ** 2
            if k % 16 == 15 and float(new) < stop:
                break
            d = r + (new / rr) * d
            rr = new
        return x


def _planes(v, kind):
    """Exact values laid out as a field of this kind: planes, or values over
    the site's largest component and that component."""
    if kind == "f64":
        return torch.view_as_real(v.transpose(0, 1).contiguous()).reshape(-1)
    f = torch.view_as_real(v.contiguous()).reshape(-1, 6)
    if kind == "f32":
        return torch.cat([f[:, :4].reshape(-1), f[:, 4:].reshape(-1)])
    scale = f.abs().amax(-1)
    return [f / scale[:, None], scale]


def _rounded(case, chi):
    """The canonical field as the packed input holds it: what the operators are given."""
    kind = case["prec"]
    if kind == "f64":
        return chi
    f = torch.view_as_real(chi.contiguous()).float()
    if kind != "f32":
        half = torch.float16 if kind == "f16" else torch.bfloat16
        s = f.abs().amax((-2, -1), keepdim=True)
        f = (f * (1.0 / s)).to(half).float() * s
    return torch.view_as_complex(f.double().contiguous())


def exact(case, seed):
    op, kind = case["op"], case["prec"]
    out = []
    for dims, u, chi in _drawn(case, seed):
        plain = _Plain(dims, u)
        del u
        if op in ("dslash", "group"):
            out.append(_planes(plain.dslash(0, _rounded(case, chi[0])), kind))
        elif op == "a_dot":
            d = _rounded(case, chi[0])
            q = plain.a(case["mass"], d)
            return [_planes(q, kind), (d.conj() * q).sum().real.reshape(1)]
        elif op == "a_mrhs":
            return [torch.cat([_planes(plain.a(m, _rounded(case, c)), kind)
                               for m, c in zip(_masses(case), chi)])]
        elif op == "solve":
            return plain.solve(case["mass"], chi[0])[None]
        else:
            return torch.stack([plain.solve(m, c) for m, c in zip(_masses(case), chi)])
    return out
