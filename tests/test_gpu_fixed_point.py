"""The fixed-point arithmetic of the FP64 volume kernel (KG and Pirozzoli fluxes) and lifting where its
scales can go wrong: flows at rest and at extreme Mach numbers, viscous fluxes above and far below the advective
ones or none at all (the lifting's general path), units far from 1, and elements whose values span too much for one scale (the kernel's general
FP64 path), at every degree parity and with ragged element counts per block. The bound is the normwise one
of the other FP64 parity tests, ULP_FACTOR times the oracle's own spread under one-ulp perturbations of its
inputs (tests/helpers.py); their flux scale holds the advective flux only, which is not the largest term here.
"""
import numpy as np
import pytest

from helpers import ULP_FACTOR, per_var_max, rounding_errors, ulp_spread
from paper_2306_12891_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(oracle_mod):
    import torch

    from paper_2306_12891_gb300 import build, dg

    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    dg.lib()
    return dg, oracle_mod, torch


def _map(x, y, z):
    return (x + 0.1 * np.sin(y) * np.cos(z), y + 0.1 * np.sin(z) * np.sin(x), z + 0.1 * np.sin(x) * np.cos(y))


def _fields(xyz, seed, mach):
    """rho, velocity and p of O(1) variation at the given Mach number (p = 1 / gamma)."""
    x, y, z = xyz[:, 0], xyz[:, 1], xyz[:, 2]
    r = np.random.default_rng(seed)
    a = r.uniform(0, 6, 5)
    rho = 1.0 + 0.2 * np.sin(x + a[0]) * np.cos(y)
    vel = [mach * np.sin(x + y + a[1]), mach * np.cos(y + z + a[2]), mach * 0.5 * np.sin(z + a[3])]
    p = (1.0 + 0.2 * np.cos(x - z + a[4])) / 1.4
    return rho, vel, p


STATES = ["rest", "mach_1e-6", "mach_1", "mach_30", "viscous", "mu_0", "units", "range_ok", "range_general"]


def _state(kind, xyz, N):
    mach = {"rest": 0.0, "mach_1e-6": 1e-6, "mach_30": 30.0}.get(kind, 0.5)
    rho, vel, p = _fields(xyz, N, mach)
    mu = {"viscous": 50.0, "rest": 0.1, "mu_0": 0.0}.get(kind, 1e-3)
    if kind == "units":
        rho, p, mu = 1e-9 * rho, 1e5 * p, 1e-12
        vel = [1e6 * v for v in vel]
    if kind in ("range_ok", "range_general"):  # one corner of the box is thin: max / min of rho and p
        ratio = 100.0 if kind == "range_ok" else 3000.0
        dip = ratio ** -np.exp(-((xyz[:, 0] - 1) ** 2 + (xyz[:, 1] - 1) ** 2 + (xyz[:, 2] - 1) ** 2))
        rho, p = rho * dip, p * dip ** 0.9  # (another exponent: equal wave speeds on both sides would tie LLF's max)
    return W.cons_from_prim(rho, *vel, p), mu


@pytest.mark.parametrize("kind", STATES)
@pytest.mark.parametrize("N,nel,vf", [(1, (5, 2, 1), "pirozzoli"), (2, (3, 1, 1), "kg"), (3, (3, 1, 1), "pirozzoli"),
                                      (4, (2, 1, 1), "kg"), (5, (3, 1, 1), "pirozzoli"), (6, (1, 2, 1), "pirozzoli"), (7, (2, 1, 1), "kg")])
def test_fixed_point_volume_terms(env, kind, N, nel, vf):
    dg, orc, torch = env
    xyz, faces = W.box_mesh(N, nel, mapping=_map)
    U0, mu = _state(kind, xyz, N)
    phys = dict(equations="ns", vflux=vf, sflux="llf", mu=mu)
    gpu, ref = dg.DG(N, xyz, faces, **phys), orc.Oracle(N, xyz, faces, **phys)
    Ut = gpu.rhs(torch.from_numpy(U0).cuda()).cpu().numpy()
    gpu.check()
    spread, Ur = ulp_spread(lambda X, V: orc.Oracle(N, X, faces, **phys).rhs(V), xyz, U0, base=ref.rhs(U0))
    err = per_var_max(Ut - Ur)
    print(f"FIXED-POINT {kind} N={N} {vf}: error / bound {err / np.maximum(ULP_FACTOR * spread, 1e-300)}")
    assert (err <= ULP_FACTOR * spread).all(), (err, ULP_FACTOR * spread)


def _stretched(N, ar, curved):
    """Two elements (N = 2: 16) with the z-edge ar times shorter than the others (x-edge: half the y-edge), and a shear layer across it:
    Mach 0.3 along x, spanwise and wall-normal velocities 10^-3 of it, or the same size (curved meshes)."""
    def wave(x, y, z):
        return x + 0.1 * np.sin(y), y + 0.1 * np.sin(x), z + 0.1 / ar * np.sin(x) * np.cos(y)
    xyz, faces = W.box_mesh(N, (2, 1, 1) if N > 2 else (4, 2, 2), hi=(W.TWO_PI, W.TWO_PI, W.TWO_PI / ar), mapping=wave if curved else None)
    x, y, z = xyz[:, 0], xyz[:, 1], ar * xyz[:, 2]
    e = 0.3 if curved else 3e-4
    rho = 1.0 + 0.1 * np.sin(z + 1.0) * np.cos(x)
    p = (1.0 + 0.05 * np.cos(x - y) * np.sin(z)) / 1.4
    vel = [0.3 * np.sin(z / 2 + 0.3) * (1 + 0.2 * np.cos(x)), e * np.cos(z + y), e * np.sin(x + y) * np.sin(z / 2) ** 2]
    return xyz, faces, W.cons_from_prim(rho, *vel, p)


@pytest.mark.parametrize("curved", [False, True])
@pytest.mark.parametrize("ar", [1, 7, 64, 1024, 16384])
@pytest.mark.parametrize("N,vf,eq,mu", [(2, "kg", "euler", 0.0), (3, "pirozzoli", "euler", 0.0), (5, "kg", "ns", 0.01),
                                        (7, "pirozzoli", "ns", 1e-3), (7, "kg", "euler", 0.0)])
def test_stretched_elements_round_no_more_than_fp64(env, ar, N, vf, eq, mu, curved):
    """The rounding error of each variable against that of the kernels' FP64 path: density, momentum, energy and mu in units
    2^350 times larger take it, and change no significand. Both are rms values over at least 50 entries of a few hundred
    roundings each: of the same size (0.5 to 1.3) where the arithmetic resolves the same."""
    dg, orc, torch = env
    xyz, faces, U = _stretched(N, ar, curved)
    out = []
    for k in (0, -350):
        phys = dict(equations=eq, vflux=vf, sflux="llf", mu=float(np.ldexp(mu, k)))
        s = dg.DG(N, xyz, faces, **phys)
        out.append(np.ldexp(s.rhs(torch.from_numpy(np.ldexp(U, k)).cuda()).cpu().numpy(), -k))
        s.check()
    Ja, J = (t.cpu().numpy() for t in s.metrics())
    here, plain = rounding_errors(orc, N, xyz, faces, U, Ja, J, out, eq, vf, "llf", mu)
    print(f"FIXED-POINT stretched {ar} curved={curved} N={N} {vf} {eq}: error / FP64 path's {np.round(here / plain, 2)}")
    assert (here <= 1.5 * plain).all(), here / plain


@pytest.mark.parametrize("N,ar", [(2, 64), (5, 1024)])
def test_stretched_elements_vjp_takes_the_fp64_path(env, N, ar):
    """The product is linear in the cotangent, and FP64 arithmetic commutes with a power of two: equal bits."""
    dg, orc, torch = env
    xyz, faces, U = _stretched(N, ar, True)
    s = dg.DG(N, xyz, faces, equations="euler", vflux="pirozzoli", sflux="llf")
    lam = np.random.default_rng(N).standard_normal(U.shape)
    a, b = (s.rhs_vjp(torch.from_numpy(U).cuda(), torch.from_numpy(np.ldexp(lam, k)).cuda()).cpu().numpy() for k in (0, 300))
    np.testing.assert_array_equal(a, np.ldexp(b, -300))


def _time(torch, call, k=20):
    for _ in range(3):
        call()
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    a.record()
    for _ in range(k):
        call()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / k


def test_elements_of_the_fp64_path_form_each_pair_once(env):
    """A right-hand side and a vector-Jacobian product with rho spanning 10^4 in every element against the same with none,
    N = 7: 2.9 and 2.1 times the time when each pair is formed once in FP64, 4.4 and 3.0 times when both nodes form it."""
    dg, orc, torch = env
    xyz, faces = W.box_mesh(7, (10, 10, 10))
    s = dg.DG(7, xyz, faces, equations="euler", vflux="pirozzoli", sflux="roe")
    lam = torch.randn(xyz.shape[0], 5, 8, 8, 8, dtype=torch.float64, device="cuda")
    times = []
    for ratio in (1.0, 1e4):
        k = np.arange(8)
        dip = ratio ** -((k[:, None, None] + k[:, None] + k) / 21.0) * np.ones_like(xyz[:, 0])
        vel = [0.1 * np.sin(xyz[:, (c + 1) % 3]) for c in range(3)]
        U = torch.from_numpy(W.cons_from_prim(dip, *vel, dip ** 0.9)).cuda()
        times.append((_time(torch, lambda: s.rhs(U)), _time(torch, lambda: s.rhs_vjp(U, lam))))
    s.check()
    r = [times[1][i] / times[0][i] for i in (0, 1)]
    print(f"FIXED-POINT FP64 path / fixed point, N = 7, 10^3: right-hand side x{r[0]:.2f}, product x{r[1]:.2f}")
    assert r[0] < 3.5 and r[1] < 2.55


@pytest.mark.parametrize("N,nel,tiny", [(1, (24, 24, 24), 0.0), (2, (16, 16, 16), 0.0), (3, (16, 16, 16), 5e-324), (7, (8, 8, 8), 0.0)])
def test_elements_without_a_cotangent(env, N, nel, tiny):
    """A product with a cotangent in one element, zero elsewhere: the FP64 path's result (the cotangent scaled by 2^900; bound
    as for the viscous sweeps below), exact zeros away from the element's neighbours, and no slower than a dense one (1.2 to
    2.2 times its time where zeros take the FP64 path). Subnormal cotangents are not zero: equal to a dense one's sum."""
    dg, orc, torch = env
    xyz, faces = W.box_mesh(N, nel, mapping=_map)
    s = dg.DG(N, xyz, faces, equations="euler", vflux="kg", sflux="llf")
    U, _ = _state("mach_1", xyz, N)
    Ud = torch.from_numpy(U).cuda()
    dense = np.random.default_rng(N).standard_normal(U.shape)
    one = np.zeros_like(U)
    one[5] = dense[5]
    Ld, Lo = (torch.from_numpy(x).cuda() for x in (dense, one))
    got, ref = (np.ldexp(s.rhs_vjp(Ud, torch.from_numpy(np.ldexp(one, k)).cuda()).cpu().numpy(), -k) for k in (0, 900))
    scl = np.abs(ref).max(axis=(0, 2, 3, 4)).reshape(1, 5, 1, 1, 1)
    assert (np.abs(got - ref) <= 1e-12 * scl).all()
    touched = {5} | {int(x) for f in faces if 5 in (f[0], f[2]) for x in (f[0], f[2])}
    far = [e for e in range(U.shape[0]) if e not in touched]
    assert (got[far] == 0.0).all()
    if tiny:  # |entry| of the product <= sum over ~100 |terms| of the operator (entries below 10^4) times tiny
        small = s.rhs_vjp(Ud, torch.full_like(Ud, tiny)).cpu().numpy()
        assert (small != 0.0).any() and np.abs(small).max() <= 1e6 * tiny
    a, b = (_time(torch, lambda x=x: s.rhs_vjp(Ud, x)) for x in (Ld, Lo))
    print(f"FIXED-POINT N={N}: product with one element's cotangent / dense: x{b / a:.2f}")
    assert b < 1.1 * a


@pytest.mark.parametrize("N", [1, 2, 3, 5])
def test_nonfinite_values_pass_through_and_are_flagged(env, N):
    """A NaN stays in its element and, at N = 1 (all nodes lie on faces), the elements that share a face with it, and dg_check
    reports it. At N = 1 and 2 a block holds 8 and 2 elements; 45 leave a ragged last one."""
    dg, orc, torch = env
    xyz, faces = W.box_mesh(N, (5, 3, 3))
    s = dg.DG(N, xyz, faces, equations="euler", vflux="pirozzoli", sflux="llf")
    U = torch.from_numpy(W.random_smooth_state(xyz, seed=N, amp=0.1)).cuda()
    clean = s.rhs(U).cpu()
    s.check()
    U[0, 4, 1, 1, 1] = float("nan")
    Ut = s.rhs(U).cpu()
    with pytest.raises(dg.DGError):
        s.check()
    assert torch.isnan(Ut[0]).any()
    reached = {0} | {int(x) for f in faces if N == 1 and 0 in (f[0], f[2]) for x in (f[0], f[2])}
    rest = [e for e in range(len(Ut)) if e not in reached]
    # elements are grouped per block: the block's others take the general path, equal to rounding
    assert torch.allclose(Ut[rest], clean[rest], rtol=0, atol=1e-11 * float(clean.abs().max()))


@pytest.mark.parametrize("kind,lam_scale", [("mach_1e-6", (1, 1, 1, 1, 1)), ("mach_30", (1, 1, 1, 1, 1)), ("mach_1", (0, 0, 0, 0, 1)),
                                            ("mach_1", (1e-20, 1, 1, 1, 1e20)), ("units", (1, 1, 1, 1, 1)),
                                            ("range_ok", (1, 1, 1, 1, 0)), ("range_general", (1, 1, 1, 1, 1))])
@pytest.mark.parametrize("N,nel,vf", [(1, (5, 2, 1), "kg"), (4, (2, 1, 1), "pirozzoli"), (7, (1, 1, 1), "kg")])
def test_fixed_point_adjoint_volume_terms(env, kind, lam_scale, N, nel, vf):
    """The adjoint volume kernel at the same scales, and with cotangents of very different sizes per variable:
    sampled entries against the oracle's complex-step columns, within 1e-12 of each variable's sum of |terms|."""
    dg, orc, torch = env
    xyz, faces = W.box_mesh(N, nel, mapping=_map)
    U, _ = _state(kind, xyz, N)
    phys = dict(equations="euler", vflux=vf, sflux="llf")
    lam = np.random.default_rng(N).standard_normal(U.shape) * np.reshape(lam_scale, (1, 5, 1, 1, 1))
    gpu = dg.DG(N, xyz, faces, **phys)
    got = gpu.rhs_vjp(torch.from_numpy(U).cuda(), torch.from_numpy(lam).cuda()).cpu().numpy().reshape(-1)
    gpu.check()
    oc = orc.Oracle(N, xyz, faces, complex_step=True, **phys)
    cols = np.random.default_rng(7).choice(U.size, 60, replace=False)
    var = (cols // U[0, 0].size) % 5
    err, scl = np.zeros(5), np.zeros(5)
    for j, v in zip(cols, var):
        Z = U.astype(np.complex128)
        Z.reshape(-1)[j] += 1e-30j
        col = oc.rhs(Z).imag / 1e-30
        err[v] = max(err[v], abs(got[j] - (col * lam).sum()))
        scl[v] = max(scl[v], (np.abs(col) * np.abs(lam)).sum())
    print(f"FIXED-POINT-ADJ {kind} {lam_scale} N={N} {vf}: {err / np.maximum(scl, 1e-300)}")
    assert (err <= 1e-12 * scl).all(), (err, scl)


@pytest.mark.parametrize("N,nel", [(1, (5, 3, 3)), (2, (3, 3, 1)), (3, (3, 1, 1)), (4, (2, 1, 1)), (5, (2, 1, 1)), (6, (1, 1, 1)),
                                   (7, (2, 1, 1))])
def test_adjoint_viscous_fixed_point_against_its_fp64_path(env, N, nel):
    """The vector-Jacobian product is linear in the cotangent: scaled by 2^900 or 2^-930 it takes the FP64 path, and must
    agree with the fixed-point result (cotangents everywhere, of energy only, and at one node) scaled alike. Fewer than
    200 roundings lie on the way to an entry, and the sum of its |terms| is below 20 times the largest entry of its
    variable: 200 x 20 x 2^-53 < 1e-12. A NaN reaches two elements far (the neighbours' viscous flux, theirs by the lifting)."""
    dg, orc, torch = env
    xyz, faces = W.box_mesh(N, nel, mapping=_map)
    U, _ = _state("mach_1", xyz, N)
    gpu = dg.DG(N, xyz, faces, equations="ns", vflux="pirozzoli", sflux="roe", mu=0.02)
    Ud = torch.from_numpy(U).cuda()
    rnd = np.random.default_rng(N).standard_normal(U.shape)
    energy = rnd * np.reshape([0, 0, 0, 0, 1.0], (1, 5, 1, 1, 1))
    point = np.zeros_like(U)
    point[-1, 1:, N, 0, N // 2] = [1.0, -0.5, 1e-3, 1e-6]
    for lam in (rnd, energy, point):
        got = gpu.rhs_vjp(Ud, torch.from_numpy(lam).cuda()).cpu().numpy()
        scl = np.abs(got).max(axis=(0, 2, 3, 4)).reshape(1, 5, 1, 1, 1)
        for k in (900, -930):
            ref = gpu.rhs_vjp(Ud, torch.from_numpy(np.ldexp(lam, k)).cuda()).cpu().numpy()
            err = np.abs(np.ldexp(ref, -k) - got) / scl
            assert err.max() <= 1e-12, (k, err.max(axis=(0, 2, 3, 4)))
    gpu.check()
    if nel[0] >= 5:  # (periodic: elements (2, 1, 0) and (3, 1, 0) are three steps away from element 0; a block's
        # elements take the FP64 path together in the volume kernel: the same bound, not the same bits)
        lam = rnd.copy()
        lam[0, 2, 0, 0, 0] = np.nan
        bad = gpu.rhs_vjp(Ud, torch.from_numpy(lam).cuda()).cpu().numpy()
        good = gpu.rhs_vjp(Ud, torch.from_numpy(rnd).cuda()).cpu().numpy()
        scl = np.abs(good).max(axis=(0, 2, 3, 4)).reshape(1, 5, 1, 1, 1)
        assert np.isnan(bad[0]).any() and (np.abs(bad[7:9] - good[7:9]) <= 1e-12 * scl).all()
