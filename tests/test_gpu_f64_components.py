"""FP64 half-pass, component by component, where the real components of a field
differ in scale by up to 2^-70 and the links hardly mix the colours: each
component has to be right relative to its own terms, not to the largest
neighbour.

Reference: the hop sum in extended precision (numpy longdouble).  Bound, with
S = sum |U_ab| |v_b| over the 48 real products of a component: 48 FMAs err by
up to 48 2^-53 S; the integer path by up to 3.9 2^-53 M and one rounding, and
is taken only where M <= 12 S: 48 2^-53 S in all.  A 12-real link's row 2 is
rebuilt: in FP64 each entry errs by up to 4 2^-53 of its products' sizes (G);
in integers by up to 3.5 2^-57, which raises 62 2^-57 M to 154 2^-57 M, 116
2^-53 S.  Where the path was integer the error is below the S terms, elsewhere
below 48 2^-53 S and the G term.
"""
import numpy as np
import pytest
import torch

import gen
import paper_1111_0125_gb300 as stg
from lattice_util import site_coords

pytestmark = pytest.mark.gpu

DIMS = (4, 6, 2, 8)


def _products(u, v):
    """(sum of u v per row, S of the real and of the imaginary part)."""
    ur, ui, vr, vi = np.abs(u.real), np.abs(u.imag), np.abs(v.real)[:, None, :], np.abs(v.imag)[:, None, :]
    return (u * v[:, None, :]).sum(-1), (ur * vr + ui * vi).sum(-1), (ur * vi + ui * vr).sum(-1)


def _reference(dims, U, chi, parity, recon):
    L = np.asarray(dims)
    U = U.astype(np.clongdouble)
    G = np.zeros(U.shape)
    if recon == 12:  # the links that such a handle holds: row 2 from rows 0 and 1
        a, b = U[..., 0, :], U[..., 1, :]
        U = U.copy()
        for k in range(3):
            p, q = (k + 1) % 3, (k + 2) % 3
            U[..., 2, k] = np.conj(a[..., p] * b[..., q] - a[..., q] * b[..., p])
            size = lambda z: np.abs(z.real) + np.abs(z.imag)
            G[..., 2, k] = (size(a[..., p]) * size(b[..., q]) + size(a[..., q]) * size(b[..., p])).astype(float)
    full = np.zeros((dims[3], dims[2], dims[1], dims[0], 3), dtype=np.clongdouble)
    c = site_coords(dims, 1 - parity)
    full[c[:, 3], c[:, 2], c[:, 1], c[:, 0]] = chi
    x = site_coords(dims, parity)
    out = np.zeros((len(x), 3), dtype=np.clongdouble)
    s_re, s_im, g_v = (np.zeros((len(x), 3)) for _ in range(3))
    for mu in range(4):
        eta = (-1.0) ** x[:, :mu].sum(axis=1)
        for way in (1, -1):
            y = x.copy()
            y[:, mu] = (x[:, mu] + way) % L[mu]
            at = x if way > 0 else y
            u = U[at[:, 3], at[:, 2], at[:, 1], at[:, 0], mu]
            g = G[at[:, 3], at[:, 2], at[:, 1], at[:, 0], mu]
            if way < 0:
                u, g = -np.conj(np.swapaxes(u, 1, 2)), np.swapaxes(g, 1, 2)
            s = eta.copy()
            if mu == 3:
                s[x[:, 3] == (L[3] - 1 if way > 0 else 0)] *= -1
            v = full[y[:, 3], y[:, 2], y[:, 1], y[:, 0]]
            d, re, im = _products(u, v)
            out += s[:, None] * d
            s_re += re.astype(float)
            s_im += im.astype(float)
            g_v += (g * (np.abs(v.real) + np.abs(v.imag)).astype(float)[:, None, :]).sum(-1)
    return out, s_re, s_im, g_v


def _links(kind):
    if kind == "unit":
        return gen.unit_gauge(DIMS)
    if kind == "phases":  # diagonal SU(3): the colours do not mix at all
        t = np.random.default_rng(1).uniform(0, 2 * np.pi, (*gen.unit_gauge(DIMS).shape[:-2], 2))
        U = np.zeros((*t.shape[:-1], 3, 3), dtype=np.complex128)
        U[..., 0, 0], U[..., 1, 1] = np.exp(1j * t[..., 0]), np.exp(1j * t[..., 1])
        U[..., 2, 2] = np.exp(-1j * (t[..., 0] + t[..., 1]))
        return U
    return gen.gauge_field(DIMS, "exp", seed=2, eps={"cold": 1e-9, "cool": 1e-3, "rough": 0.5}[kind])


@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("kind", ["unit", "phases", "cold", "cool", "rough"])
@pytest.mark.parametrize("bits", [(0, 0, 0, 0), (0, 5, 10, 0), (0, 33, 60, 0), (70, 0, 3, 0), (0, 0, 0, 40)])
def test_components_at_different_scales(kind, bits, recon):
    """Colours times 2^-bits, imaginary parts times 2^-bits[3]."""
    U = _links(kind)
    chi = gen.source(DIMS, seed=5) * 2.0 ** -np.asarray(bits[:3])
    chi = chi.real + 1j * (chi.imag * 2.0 ** -bits[3])
    s_bound, g_bound = (48 * 2.0 ** -53, 0.0) if recon == 18 else (116 * 2.0 ** -53, 4 * 2.0 ** -53)
    with stg.Gauge(DIMS, U, sloppy=stg.STG_FP64, recon=recon) as h:
        for parity in (0, 1):
            want, s_re, s_im, g_v = _reference(DIMS, U, chi, parity, recon)
            f = h.pack(torch.from_numpy(chi).cuda(), stg.STG_FP64)
            got = h.unpack(h.dslash(f, parity, stg.STG_FP64), stg.STG_FP64).cpu().numpy()
            for err, s in (((got.real - want.real), s_re), ((got.imag - want.imag), s_im)):
                assert np.all(np.abs(err).astype(float) <= s_bound * s + g_bound * g_v)
