"""The FP64 Dslash on limb links (csrc/fix64.cuh) where it can go wrong:
scales of the field over the whole FP64 range, spreads inside one
neighbourhood, zero / non-finite sites, and links that keep doubles.

Reference: the hop sum in extended precision (numpy longdouble, at least 64
significand bits).  Bound per component, from the number formats, with v the
largest component among the eight neighbours: cutting the neighbours to 57
bits 2^-56 v per product, at most 8 sqrt(6) < 20 of them after unitarity
(2^-51.6 v); links to 2^-57, 48 products (2^-51.4 v); the omitted low products
48 2^-59 v (2^-53.4 v); one rounding of a value below 20 v (2^-48.7 v).  The
sum is below 2^-48 v.
"""
import numpy as np
import pytest
import torch

import gen
import paper_1111_0125_gb300 as stg
from lattice_util import site_coords

pytestmark = pytest.mark.gpu

DIMS = (4, 6, 2, 8)
BOUND = 2.0 ** -48


def _reference(dims, U, chi, parity):
    """(D chi on the sites of parity, largest neighbour component per site)."""
    L = np.asarray(dims)
    full = np.zeros((dims[3], dims[2], dims[1], dims[0], 3), dtype=np.clongdouble)
    c = site_coords(dims, 1 - parity)
    full[c[:, 3], c[:, 2], c[:, 1], c[:, 0]] = chi
    U = U.astype(np.clongdouble)
    x = site_coords(dims, parity)
    out = np.zeros((len(x), 3), dtype=np.clongdouble)
    big = np.zeros(len(x))
    for mu in range(4):
        eta = (-1.0) ** x[:, :mu].sum(axis=1)
        for way in (1, -1):
            y = x.copy()
            y[:, mu] = (x[:, mu] + way) % L[mu]
            at = x if way > 0 else y
            u = U[at[:, 3], at[:, 2], at[:, 1], at[:, 0], mu]
            s = eta.copy()
            if mu == 3:
                s[x[:, 3] == (L[3] - 1 if way > 0 else 0)] *= -1
            v = full[y[:, 3], y[:, 2], y[:, 1], y[:, 0]]
            if way > 0:
                out += s[:, None] * (u * v[:, None, :]).sum(-1)
            else:
                out -= s[:, None] * (np.conj(np.swapaxes(u, 1, 2)) * v[:, None, :]).sum(-1)
            big = np.maximum(big, np.maximum(np.abs(v.real), np.abs(v.imag)).max(-1).astype(float))
    return out, big


def _dslash(g, chi, parity):
    f = g.pack(torch.from_numpy(chi).cuda(), stg.STG_FP64)
    return g.unpack(g.dslash(f, parity, stg.STG_FP64), stg.STG_FP64).cpu().numpy()


def _check(got, want, big, bound=BOUND):
    d = np.abs(got - want).astype(float)
    assert np.all(d <= bound * big[:, None]), float((d / np.maximum(big, 1e-320)[:, None]).max())


@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("scale", [2.0 ** -1060, 2.0 ** -900, 2.0 ** -880, 1e-20, 1.0, 1e20, 2.0 ** 1000,
                                   2.0 ** 1015])
@pytest.mark.parametrize("spread", [0, 40, 80])
def test_field_scales(recon, scale, spread):
    """Every site times a power of two of its own within 2^-spread .. 1."""
    U = gen.gauge_field(DIMS, "haar", seed=3)
    chi = gen.source(DIMS, seed=5)
    if spread:
        chi = chi * 2.0 ** -np.random.default_rng(7).integers(0, spread, (len(chi), 1))
    chi = chi * scale
    with stg.Gauge(DIMS, U, sloppy=stg.STG_FP64, recon=recon) as g:
        for parity in (0, 1):
            want, big = _reference(DIMS, U, chi, parity)
            got = _dslash(g, chi, parity)
            # below 2^-1022 results are rounded to the subnormal grid
            tiny = 2.0 ** -1068
            d = np.abs(got - want).astype(np.longdouble)
            assert np.all(d <= BOUND * big[:, None].astype(np.longdouble) + tiny)


@pytest.mark.parametrize("recon", [18, 12])
def test_zero_point_and_non_finite(recon):
    U = gen.gauge_field(DIMS, "exp", seed=2, eps=0.4)
    vh = int(np.prod(DIMS)) // 2
    with stg.Gauge(DIMS, U, sloppy=stg.STG_FP64, recon=recon) as g:
        assert not np.any(_dslash(g, np.zeros((vh, 3), dtype=np.complex128), 0))
        point = np.zeros((vh, 3), dtype=np.complex128)
        point[vh // 3, 1] = 0.7 - 0.2j
        want, big = _reference(DIMS, U, point, 0)
        got = _dslash(g, point, 0)
        _check(got, want, big)
        assert not np.any(got[big == 0.0])
        for bad in (np.inf, np.nan):
            chi = gen.source(DIMS, seed=6)
            clean, big = _reference(DIMS, U, chi, 0)
            chi[vh // 3, 2] = bad
            touched = _reference(DIMS, U, point, 0)[1] > 0.0
            got = _dslash(g, chi, 0)
            assert not np.any(np.isfinite(got[touched]).all(axis=1))
            _check(got[~touched], clean[~touched], big[~touched])


def test_unit_links_and_links_that_are_not_unitary():
    """Entries of exactly 1 and 0 (limb 2^29); links scaled by 1.5 keep the
    FP64 arithmetic (bound: 48 roundings of at most 1.5 sqrt(6) 8 v)."""
    chi = gen.source(DIMS, seed=8)
    for U, bound in ((gen.unit_gauge(DIMS), BOUND), (1.5 * gen.gauge_field(DIMS, "haar", seed=4), 48 * 30 * 2.0 ** -53)):
        with stg.Gauge(DIMS, U, sloppy=stg.STG_FP64, recon=18) as g:
            for parity in (0, 1):
                want, big = _reference(DIMS, U, chi, parity)
                _check(_dslash(g, chi, parity), want, big, bound)


def test_error_is_not_above_the_fp64_arithmetic():
    """On Gaussian fields the norm-wise error stays below that of 48 FP64 FMAs
    in sequence, 3e-16 measured; the integer form rounds once (2^-53 / sqrt(3)
    and the cuts)."""
    U = gen.gauge_field(DIMS, "exp", seed=1, eps=0.5)
    chi = gen.source(DIMS, seed=9)
    with stg.Gauge(DIMS, U, sloppy=stg.STG_FP64, recon=18) as g:
        want, _ = _reference(DIMS, U, chi, 0)
        d = (_dslash(g, chi, 0) - want).astype(np.complex128)
    assert np.linalg.norm(d) <= 2.0 ** -53 * np.linalg.norm(want.astype(np.complex128))
