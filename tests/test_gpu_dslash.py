"""GPU Dslash and normal operator vs the FP64 CPU oracle, through the C ABI.

Bars (fixed by the build's target): relative L2 error <= 1e-12 for the FP64
Dslash and <= 1e-5 for the FP32 Dslash, element by element on seeded inputs.
Small lattices cover several thread blocks and a ragged tail (Vh not a
multiple of the 128-thread block); 32^4 (the single-mass benchmark lattice,
in the launch configuration the benchmark times) is checked on sampled sites
the oracle computes one by one, plus the free-field closed form at every site.
"""

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-5}  # F64, F32


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def fold_phases(L, U, hop, apbc):
    """Multiply links by eta_mu(n) and the boundary sign (test-side, for PHASES_FOLDED)."""
    c = synth.site_coords(L)
    out = U.copy()
    for mu in range(4):
        s = np.where(c[:, :mu].sum(axis=1) % 2 == 0, 1.0, -1.0) if mu else np.ones(len(c))
        if mu == 3 and apbc:
            s = np.where(c[:, 3] + hop >= L[3], -s, s)
        out[:, mu] *= s[:, None, None]
    return out


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (8, 8, 8, 8), (6, 8, 10, 12), (8, 10, 12, 14)])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("recon", [False, True])
def test_dslash_matches_oracle(sqcg, links_cache, L, prec, recon):
    fat, lng = links_cache(L, 1001)
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng, recon12=recon)
        for out_par in (0, 1):
            psi = synth.gaussian_source(L, 2000 + out_par)
            d_in = lat.pack(psi, prec)
            d_out = lat.new_spinor(prec)
            lat.dslash(out_par, d_in, d_out, prec)
            got = lat.unpack(d_out, prec)
            want = oracle.dslash(L, fat, lng, psi, out_par)
            assert rel(got, want) <= TOL[prec], (L, prec, recon, out_par, rel(got, want))


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (6, 8, 10, 12)])
@pytest.mark.parametrize("recon", [False, True])
@pytest.mark.parametrize("apbc", [False, True])
def test_dslash_eight_way_matches_oracle(sqcg, links_cache, L, recon, apbc):
    """8-way FP32 storage (backward links at the site that uses them) gives the same D."""
    fat, lng = links_cache(L, 1001)
    with sqcg.Lattice(L, antiperiodic_t=apbc) as lat:
        lat.load_links(fat, lng, recon12=recon, eight_way=True)
        for out_par in (0, 1):
            psi = synth.gaussian_source(L, 2000 + out_par)
            out = lat.new_spinor(1)
            lat.dslash(out_par, lat.pack(psi, 1), out, 1)
            want = oracle.dslash(L, fat, lng, psi, out_par, apbc)
            assert rel(lat.unpack(out, 1), want) <= TOL[1]
        # FP64 stays forward-only and exact
        out = lat.new_spinor(0)
        psi = synth.gaussian_source(L, 3)
        lat.dslash(0, lat.pack(psi), out)
        assert rel(lat.unpack(out), oracle.dslash(L, fat, lng, psi, 0, apbc)) <= TOL[0]


@pytest.mark.parametrize("apbc", [False, True])
def test_dslash_periodic_and_folded_phases(sqcg, links_cache, apbc):
    L = (6, 8, 10, 12)
    fat, lng = links_cache(L, 77)
    psi = synth.gaussian_source(L, 5)
    want = oracle.dslash(L, fat, lng, psi, 1, antiperiodic_t=apbc)
    with sqcg.Lattice(L, antiperiodic_t=apbc) as lat:
        lat.load_links(fat, lng)
        out = lat.new_spinor(0)
        lat.dslash(1, lat.pack(psi), out)
        assert rel(lat.unpack(out), want) <= 1e-12
    # the caller folds the phases itself
    with sqcg.Lattice(L, antiperiodic_t=apbc, phases_folded=True) as lat:
        lat.load_links(fold_phases(L, fat, 1, apbc), fold_phases(L, lng, 3, apbc), recon12=True)
        out = lat.new_spinor(0)
        lat.dslash(1, lat.pack(psi), out)
        assert rel(lat.unpack(out), want) <= 1e-12


def test_recon12_rejected_for_non_su3_long_links(sqcg, links_cache):
    L = (4, 4, 4, 6)
    fat, lng = links_cache(L, 3)
    bad = lng.copy()
    bad[17, 2] *= 1.001  # one link is no longer s * SU(3) with the global s
    with sqcg.Lattice(L) as lat:
        with pytest.raises(sqcg.SqcgError) as e:
            lat.load_links(fat, bad, recon12=True)
        assert e.value.name == "RECON_REJECTED"
        lat.load_links(fat, bad, recon12=False)  # full storage is always accepted


@pytest.mark.parametrize("L", [(8, 8, 8, 8), (6, 8, 10, 12)])
@pytest.mark.parametrize("prec", [0, 1])
def test_normal_op_matches_oracle(sqcg, links_cache, L, prec):
    fat, lng = links_cache(L, 1001)
    sigma = 4 * 0.1**2
    x = synth.gaussian_source(L, 2100)
    want = oracle.normal_op(L, fat, lng, sigma, x)
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng)
        y = lat.new_spinor(prec)
        lat.normal_op(sigma, lat.pack(x, prec), y, prec)
        assert rel(lat.unpack(y, prec), want) <= TOL[prec]


def test_anti_hermiticity_on_gpu(sqcg, links_cache):
    L = (16, 16, 16, 16)
    fat, lng = links_cache(L, 1001)
    y_e = synth.gaussian_source(L, 1)
    x_o = synth.gaussian_source(L, 2)
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng)
        a, b = lat.new_spinor(), lat.new_spinor()
        lat.dslash(0, lat.pack(x_o), a)
        lat.dslash(1, lat.pack(y_e), b)
        lhs = np.vdot(y_e, lat.unpack(a))
        rhs = np.vdot(lat.unpack(b), x_o)
    assert abs(lhs + rhs) <= 1e-13 * abs(lhs)


@pytest.mark.parametrize("prec", [0, 1])
def test_free_field_closed_form_32(sqcg, prec):
    """Unit links: D on a plane wave is sum_mu eta_mu 2i (c1 sin p + c3 sin 3p) times the wave, at every site."""
    L = (32, 32, 32, 32)
    c1, c3 = 0.9, -1.0 / 24.0
    fat, lng = synth.unit_links(L, c1, c3)
    k = (3, 1, 7, 5)
    colour = (0.6, -0.2 + 0.5j, 1.0j)
    psi = synth.plane_wave(L, k, 0, colour)
    p = np.array([2 * np.pi * k[m] / L[m] for m in range(3)] + [(2 * k[3] + 1) * np.pi / L[3]])
    c = synth.site_coords(L)[synth.parity_sites(L, 1)]
    coef = np.zeros(len(c), dtype=np.complex128)
    for mu in range(4):
        eta = np.where(c[:, :mu].sum(axis=1) % 2 == 0, 1.0, -1.0) if mu else np.ones(len(c))
        coef += eta * 2j * (c1 * np.sin(p[mu]) + c3 * np.sin(3 * p[mu]))
    want = coef[:, None] * synth.plane_wave(L, k, 1, colour)
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng, recon12=True)
        out = lat.new_spinor(prec)
        lat.dslash(1, lat.pack(psi, prec), out, prec)
        got = lat.unpack(out, prec)
    assert rel(got, want) <= (1e-12 if prec == 0 else 1e-5)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("recon", [False, True])
def test_dslash_32_sampled_sites(sqcg, links_cache, prec, recon):
    """Full benchmark lattice: GPU output at sampled sites (including every boundary) vs the oracle."""
    L = (32, 32, 32, 32)
    fat, lng = links_cache(L, 1002)
    psi = synth.gaussian_source(L, 2200)
    out_par = 1
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng, recon12=recon)
        out = lat.new_spinor(prec)
        lat.dslash(out_par, lat.pack(psi, prec), out, prec)
        got = lat.unpack(out, prec)
    sites = synth.parity_sites(L, out_par)
    c = synth.site_coords(L)[sites]
    rng = np.random.default_rng(0)
    edge = np.nonzero((c == 0).any(axis=1) | (c == 31).any(axis=1) | (c == 2).any(axis=1) | (c == 29).any(axis=1))[0]
    pick = np.unique(np.concatenate([rng.choice(len(sites), 600, replace=False), rng.choice(edge, 400, replace=False),
                                     [0, len(sites) - 1]]))
    want = oracle.dslash_sites(L, fat, lng, psi, 1 - out_par, sites[pick])
    assert rel(got[pick], want) <= TOL[prec]


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (8, 8, 8, 8), (6, 8, 10, 12), (8, 10, 12, 14), (16, 16, 16, 16)])
@pytest.mark.parametrize("par", [0, 1])
def test_dslash_float_float_matches_oracle(sqcg, links_cache, L, par):
    """The float-float Dslash (hi + lo floats per real, error-free products and sums on the FP32 pipe)
    against the FP64 oracle at the FP64 bar, 1e-12, on cubic and ragged lattices and both parities."""
    fat, lng = links_cache(L, 1001)
    psi = synth.gaussian_source(L, 2001 + par)
    want = oracle.dslash(L, fat, lng, psi, par)
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng, recon12=True)  # the float-float copy is always 18-real
        out = lat.new_spinor(sqcg.FF)
        lat.dslash(par, lat.pack(psi, sqcg.FF), out, sqcg.FF)
        got = lat.unpack(out, sqcg.FF)
        # and the FP64 kernel on the same input, for the record of how close the two arithmetics are
        out64 = lat.new_spinor(sqcg.F64)
        lat.dslash(par, lat.pack(psi, sqcg.F64), out64, sqcg.F64)
        got64 = lat.unpack(out64, sqcg.F64)
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    assert err <= 1e-12, err
    assert np.linalg.norm(got - got64) / np.linalg.norm(got64) <= 1e-12


def test_float_float_pack_round_trip_and_free_field(sqcg):
    """Packing splits each real into hi = fl32(v), lo = fl32(v - hi) (hi + lo = v to 2^-48 relative), and the
    float-float Dslash reproduces the free-field plane-wave eigenvalue of D to that precision."""
    L = (8, 8, 8, 8)
    c1, c3 = 0.9, -1.0 / 24.0
    fat, lng = synth.unit_links(L, c1, c3)
    psi = synth.gaussian_source(L, 77)
    with sqcg.Lattice(L) as lat:
        got = lat.unpack(lat.pack(psi, sqcg.FF), sqcg.FF)
        assert np.max(np.abs(got - psi)) <= 1e-14 * np.max(np.abs(psi))
        lat.load_links(fat, lng)
        k = (1, 2, 3, 1)
        pw = synth.plane_wave(L, k, 1, (1.0, 0.5j, -0.25))
        out = lat.new_spinor(sqcg.FF)
        lat.dslash(0, lat.pack(pw, sqcg.FF), out, sqcg.FF)
        got = lat.unpack(out, sqcg.FF)
    want = oracle.dslash(L, fat, lng, pw, 0)
    assert np.linalg.norm(got - want) / np.linalg.norm(want) <= 1e-13


# Each form of the split Dslash at a remainder of its 32-site groups (SMs: 152): 78.75 groups and a quarter of
# an SM's tile (8 warps a group in every precision), 367.5 groups (4 warps in FP64 and float-float), 600.25
# groups (4 warps in the 12-real FP32 form), and 3 tiles a SM (one thread a site for 12-real FP32).
@pytest.mark.parametrize("L", [(6, 6, 10, 14), (14, 14, 10, 12), (14, 14, 14, 14), (18, 18, 18, 20)])
@pytest.mark.parametrize("eight", [False, True])
@pytest.mark.parametrize("recon", [False, True])
def test_split_dslash_remainders(sqcg, links_cache, L, recon, eight):
    """D on both parities and the normal operator at lattice sizes on both sides of every line of the rule that
    chooses how many warps share a site's hops, against the oracle at the bars above (float-float: 1e-12)."""
    fat, lng = links_cache(L, 1003)
    psi = synth.gaussian_source(L, 2003)
    want = [oracle.dslash(L, fat, lng, psi, par) for par in (0, 1)]
    want_a = oracle.normal_op(L, fat, lng, 0.04, psi)
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng, recon12=recon, eight_way=eight)
        for prec, bar in ((0, 1e-12), (1, 1e-5), (2, 1e-12)):
            d_in, out = lat.pack(psi, prec), lat.new_spinor(prec)
            for par in (0, 1):
                lat.dslash(par, d_in, out, prec)
                assert rel(lat.unpack(out, prec), want[par]) <= bar, (prec, par)
            if prec != 2:
                lat.normal_op(0.04, d_in, out, prec)
                assert rel(lat.unpack(out, prec), want_a) <= bar, prec


# Where the rule turns by how full the last wave of one thread a site is (152 SMs): 1.90 tiles a SM (FP64: one thread),
# 5.30 (float-float: one thread; 8-way 12-real: alone one thread), 8.53 (full links: the normal operator one thread).
@pytest.mark.parametrize("L,recon,eight", [((12, 14, 20, 22), False, False), ((18, 20, 22, 26), True, True),
                                           ((24, 24, 24, 24), False, False), ((24, 24, 24, 24), True, True)])
def test_split_dslash_by_the_last_wave(sqcg, links_cache, L, recon, eight):
    fat, lng = links_cache(L, 1003)
    psi = synth.gaussian_source(L, 2003)
    want = [oracle.dslash(L, fat, lng, psi, par) for par in (0, 1)]
    want_a = oracle.normal_op(L, fat, lng, 0.04, psi)
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng, recon12=recon, eight_way=eight)
        for prec, bar in ((0, 1e-12), (1, 1e-5), (2, 1e-12)):
            d_in, out = lat.pack(psi, prec), lat.new_spinor(prec)
            for par in (0, 1):
                lat.dslash(par, d_in, out, prec)
                assert rel(lat.unpack(out, prec), want[par]) <= bar, (prec, par)
            if prec != 2:
                lat.normal_op(0.04, d_in, out, prec)
                assert rel(lat.unpack(out, prec), want_a) <= bar, prec


@pytest.mark.parametrize("where", [(0, 0), (1, 2), (-1, 3)])
@pytest.mark.parametrize("folded", [False, True])
def test_recon12_check_finds_one_link(sqcg, links_cache, where, folded):
    """The 12-real eligibility test sees a change of 1e-10 (its line is 1e-12) in any one long link: of its scale,
    of its determinant's phase, of one element. A refusal leaves the links before it in use; a change of 1e-14
    passes. 648 sites a parity: the last block of the check is partly filled."""
    L = (6, 6, 6, 6)
    fat, lng = links_cache(L, 1005)
    psi = synth.gaussian_source(L, 2005)
    want = oracle.dslash(L, fat, lng, psi, 0)
    if folded:
        fat, lng = fold_phases(L, fat, 1, True), fold_phases(L, lng, 3, True)

    def changed(kind, eps):
        out = lng.copy()
        u = out[where[0], where[1]]
        if kind == "scale":
            u *= 1 + eps
        elif kind == "phase":
            u *= np.exp(1j * eps)
        else:
            u[1, 2] += eps * np.abs(u).max()
        return out

    with sqcg.Lattice(L, phases_folded=folded) as lat:
        lat.load_links(fat, lng, recon12=True)
        out = lat.new_spinor(1)
        for kind in ("scale", "phase", "element"):
            with pytest.raises(sqcg.SqcgError) as err:
                lat.load_links(fat, changed(kind, 1e-10), recon12=True)
            assert err.value.name == "RECON_REJECTED"
            lat.dslash(0, lat.pack(psi, 1), out, 1)
            assert rel(lat.unpack(out, 1), want) <= TOL[1]
            lat.load_links(fat, changed(kind, 1e-14), recon12=True)


@pytest.mark.parametrize("power", [-300, 300])
def test_recon12_check_at_the_ends_of_the_range(sqcg, links_cache, power):
    """Long links scaled so far that the squares of their products leave the range of FP64 (their determinants do
    not): a link whose rows are not of one length, with the determinant of the others, is refused, the links themselves
    pass."""
    L = (4, 4, 4, 4)
    fat, lng = links_cache(L, 1005)
    lng = lng * 2.0 ** power
    bad = lng.copy()
    bad[5, 1] *= np.array([1 + 1e-6, 1 / (1 + 1e-6), 1])[:, None]
    with sqcg.Lattice(L) as lat:
        lat.load_links(fat, lng, recon12=True)
        with pytest.raises(sqcg.SqcgError) as err:
            lat.load_links(fat, bad, recon12=True)
        assert err.value.name == "RECON_REJECTED"


def test_links_reloaded_in_other_forms(sqcg, links_cache):
    """Links loaded again and again into one context, with other values and in every storage form (arrays of the same
    size are used again), on a lattice whose last 32-site block is half filled."""
    L = (6, 6, 6, 6)
    psi = synth.gaussian_source(L, 2006)
    with sqcg.Lattice(L) as lat:
        for k, (recon, eight) in enumerate([(False, False), (True, False), (True, True), (False, True), (True, False),
                                            (True, False), (False, False)]):
            fat, lng = links_cache(L, 1005 + k % 2)
            lat.load_links(fat, lng, recon12=recon, eight_way=eight)
            for prec, bar in ((0, 1e-12), (1, 1e-5), (2, 1e-12)):
                out = lat.new_spinor(prec)
                for par in (0, 1):
                    lat.dslash(par, lat.pack(psi, prec), out, prec)
                    want = oracle.dslash(L, fat, lng, psi, par)
                    assert rel(lat.unpack(out, prec), want) <= bar, (k, prec, par)


@pytest.mark.parametrize("recon", [False, True])
def test_links_reloaded_behind_work_on_another_stream(sqcg, links_cache, recon):
    """Operators and a pack that wait on a side stream while the default stream loads other links of the same form,
    whose arrays and staging are kept: they run on the links and the vector of their time. The side stream is held
    back by a tenth of a second, the packed vector is pinned, so that nothing of it has run when the loading starts."""
    L = (6, 8, 10, 12)
    old, new = links_cache(L, 1005), links_cache(L, 1006)
    psi = synth.gaussian_source(L, 2007)
    pinned = torch.from_numpy(synth.gaussian_source(L, 2008).view(np.float64)).pin_memory().numpy().view(np.complex128)
    side = torch.cuda.Stream()
    with sqcg.Lattice(L) as lat:
        lat.load_links(*old, recon12=recon)
        vecs = {prec: lat.pack(psi, prec) for prec in (0, 1)}
        outs = {prec: [lat.new_spinor(prec) for _ in range(20)] for prec in (0, 1)}
        packed = lat.new_spinor()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(200_000_000)
            lat.pack(pinned, out=packed)
            for prec in (0, 1):
                for out in outs[prec]:
                    lat.normal_op(0.04, vecs[prec], out, prec)
        lat.load_links(*new, recon12=recon)
        side.synchronize()
        want, want_new = (oracle.normal_op(L, *links, 0.04, psi) for links in (old, new))
        assert np.array_equal(lat.unpack(packed), pinned)
        for prec in (0, 1):
            for out in outs[prec]:
                assert rel(lat.unpack(out, prec), want) <= TOL[prec]
            lat.normal_op(0.04, vecs[prec], outs[prec][0], prec)
            assert rel(lat.unpack(outs[prec][0], prec), want_new) <= TOL[prec]
