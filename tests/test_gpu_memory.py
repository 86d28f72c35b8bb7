"""Solves under a bound on the context's workspace (host-side, as if the device had no
more memory): the further fields of a ring of directions and of a group of shifts are
taken only where everything a solve needs has its place."""
import ctypes as ct

import numpy as np
import pytest

from oracle import solvers as S
from oracle import dirac as D
from synth import fields as F
from tests.gpu_util import Lat, from_dev, to_dev

pytestmark = pytest.mark.gpu

DIMS = (8, 6, 6, 10)
VH = 8 * 6 * 6 * 10 // 2
ACT = {1: dict(mu=0.01), 2: dict(mubar=0.1246, epsbar=0.1350)}


def _field(prec, nf):
    """Bytes of a native field: 8 (FP64 and double word), 4 or 2 a real, 16-bit scales."""
    return VH * (24 * nf * {0: 8, 1: 4, 2: 2, 3: 2}[prec] + (4 if prec >= 2 else 0))


def _bound(lat, nbytes):
    f = lat.tm.lib.tmk_scratch_limit
    f.argtypes, f.restype = [ct.c_void_p, ct.c_size_t], ct.c_size_t
    return f(lat.ctx, nbytes)


def _lat(nf, seed=1500):
    u = F.gauge_field(DIMS, seed)
    return D.TwistedMassClover(u, DIMS, 0.1394, 1.69, **ACT[nf]), Lat(u, DIMS, 0.1394, 1.69, **ACT[nf])


# fields a CG solve cannot do without: x, b, r, A x and the operator's two
# intermediates in FP64, the double-word x, and r, p and two intermediates in the
# sloppy precision with x in FP32 (plain FP64: p alone, the rest serves)
def _cg_need(prec, nf):
    if prec == 0:
        return 7 * _field(0, nf)
    return 7 * _field(0, nf) + 4 * _field(prec, nf) + _field(1, nf)


@pytest.mark.parametrize("nf", [1, 2])
@pytest.mark.parametrize("prec", [0, 1, 2, 3], ids=["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("extra", [0, 1, 2, 3], ids=lambda e: f"{e} more")
def test_cg_fits_where_its_needed_fields_do(prec, nf, extra):
    """The needed fields and 0 to 3 more of a direction's size: a ring of 1, 2, 2, 4."""
    op, lat = _lat(nf)
    tm = lat.tm
    code, apply = (tm.TM_MDAGM, op.MdagM) if nf == 1 else (tm.TM_QH_SQ, op.heavy_sq)
    limit = _cg_need(prec, nf) + extra * _field(prec, nf)
    try:
        b = F.odd_spinor(DIMS, 1501, nf)
        _bound(lat, limit)
        for _ in range(2):
            x = to_dev(np.zeros_like(b))
            info = tm.tm_solve_cg(lat.ctx, code, tm.solve_params(tol=1e-9, sloppy=prec), x, to_dev(b))
            assert info.status == 0 and S.rel_residual(apply, from_dev(x, b.shape), b) <= 1.05e-9
        assert _bound(lat, limit) <= limit
        # and nothing left over that the solve had no use for
        assert _bound(lat, limit) == limit - (_field(prec, nf) if extra == 2 else 0)
    finally:
        lat.close()


@pytest.mark.parametrize("nf,ns", [(1, 2), (2, 6), (1, 16)])
@pytest.mark.parametrize("prec,refine", [(1, 1), (1, 3), (0, 1)], ids=["f32", "f32 then f16", "f64 then f32"])
def test_multishift_fits_where_its_needed_fields_do(prec, refine, nf, ns):
    """Bounded by what the multishift solve and the refinement of one shift need, the
    shifts are refined without a ring's or a group's further fields; unbounded with them.
    Both give solutions that meet the tolerance."""
    op, lat = _lat(nf)
    tm = lat.tm
    code, apply = (tm.TM_MDAGM, op.MdagM) if nf == 1 else (tm.TM_QH_SQ, op.heavy_sq)
    f64, f32, fs, fr = _field(0, nf), _field(1, nf), _field(prec, nf), _field(refine, nf)
    # x_k and b; r, p and two intermediates; p_k (and x_k in FP32); the refinement's r, A x,
    # two intermediates, double-word x in FP64, its own r and x
    need = (ns + 1) * f64 + 4 * fs + ns * fs + (ns * f32 if prec else 0) + 5 * f64 + fr + f32
    shifts = [0.01 * 1.6 ** k for k in range(ns)]
    try:
        b = F.odd_spinor(DIMS, 1502, nf)
        sp = tm.solve_params(tol=1e-9, sloppy=prec, refine=refine)
        for limit in (need, 0, need):
            _bound(lat, limit)
            xs = [to_dev(np.zeros_like(b)) for _ in shifts]
            infos = tm.tm_solve_multishift(lat.ctx, code, shifts, xs, to_dev(b), sp)
            assert all(i.status == 0 for i in infos)
            for s, x in zip(shifts, xs):
                v = from_dev(x, b.shape)
                assert np.linalg.norm(b - apply(v) - s * v) <= 1.05e-9 * np.linalg.norm(b), (limit, s)
            held = _bound(lat, limit)
            if limit == 0:
                full = held
                assert full > need
            else:   # (after the unbounded call: what it had taken, and nothing more)
                assert held <= need or held == full
    finally:
        lat.close()


def test_spare_fields_are_given_back_for_a_needed_one():
    """What a group of shifts left in the context makes room for another solve."""
    op, lat = _lat(1)
    tm = lat.tm
    try:
        b = F.odd_spinor(DIMS, 1503)
        shifts = [0.01 * 1.4 ** k for k in range(16)]
        xs = [to_dev(np.zeros_like(b)) for _ in shifts]
        tm.tm_solve_multishift(lat.ctx, tm.TM_MDAGM, shifts, xs, to_dev(b), tm.solve_params(tol=1e-9, sloppy=1))
        held = _bound(lat, 0)
        _bound(lat, held)
        x = to_dev(np.zeros_like(b))
        info = tm.tm_solve_cg(lat.ctx, tm.TM_MDAGM, tm.solve_params(tol=1e-9, sloppy=0), x, to_dev(b))
        assert info.status == 0 and S.rel_residual(op.MdagM, from_dev(x, b.shape), b) <= 1.05e-9
        assert _bound(lat, held) < held
    finally:
        lat.close()


@pytest.mark.parametrize("room", [1, 3, 8, 12, 20], ids=lambda r: f"{r} fields")
def test_multishift_without_room_returns_an_error(room):
    """A multishift or rational call whose fields do not fit says so, in the records too,
    and the context goes on working."""
    op, lat = _lat(1)
    tm = lat.tm
    try:
        b = F.odd_spinor(DIMS, 1504)
        shifts = [0.01, 0.02, 0.04, 0.08]
        _bound(lat, room * _field(0, 1))
        xs = [to_dev(np.zeros_like(b)) for _ in shifts]
        sp = tm.solve_params(tol=1e-9, sloppy=1)
        infos = tm.tm_solve_multishift(lat.ctx, tm.TM_MDAGM, shifts, xs, to_dev(b), sp, check=False)
        fits = room == 20
        assert all(i.status == (0 if fits else tm.TM_ERR_OOM) for i in infos)
        assert all((float(x.norm()) > 0) == (room >= 12) for x in xs)   # (12: the refinement had no room)
        if not fits:
            with pytest.raises(tm.TMError) as e:
                tm.tm_solve_multishift(lat.ctx, tm.TM_MDAGM, shifts, xs, to_dev(b), sp)
            assert e.value.status == tm.TM_ERR_OOM
            with pytest.raises(tm.TMError):
                tm.tm_rational_apply(lat.ctx, tm.TM_MDAGM, (1.0, [0.5] * 4, shifts), to_dev(b), to_dev(b), sp)
        _bound(lat, 0)
        infos = tm.tm_solve_multishift(lat.ctx, tm.TM_MDAGM, shifts, xs, to_dev(b), sp)
        assert all(i.status == 0 and i.true_rel_res <= 1e-9 for i in infos)
    finally:
        lat.close()
