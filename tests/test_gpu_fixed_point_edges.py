"""The integer-pipe kernels of the 2D path at the edges of what they take."""
import json

import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KB = [(1, O.BASIS_Q), (1, O.BASIS_P), (2, O.BASIS_Q), (2, O.BASIS_P), (3, O.BASIS_Q), (3, O.BASIS_P)]
SYSTEMS = [O.EULER, O.ADVECTION, O.BURGERS]


def _desc(system, k, basis, nx, ny, bx=1.0, by=1.0, bc=O.PERIODIC, rk=3, gamma=1.4):
    return dict(dim=2, nx=nx, ny=ny, k=k, basis=basis, system=system, bc=bc, oe=1, rk=rk, ax=0.0, bx=bx, ay=0.0,
                by=by, gamma=gamma, cfl=0.1, adv_x=1.0, adv_y=-0.7)


def _pair(*a, **kw):
    from paper_2503_12473_gb300 import oecdg as G
    d = _desc(*a, **kw)
    return O.Problem(**d), G.Context(G.MeshDesc(**d))


def _state(p, rng, size=0.02):
    """Coefficients of the given size about a uniform physical state."""
    u = size * rng.standard_normal(p.shape)
    u[:, :, 0] += np.array([1.0, 0.3, -0.2, 4.0] if p.nfields == 4 else [1.0])[None, :, None, None]
    if p.nxs != p.nx or p.nys != p.ny:  # the primal mesh leaves the padded slots at 0
        u[0, :, :, p.ny:] = 0.0
        u[0, :, :, :, p.nx:] = 0.0
    return u


SIDES = {"periodic": O.PERIODIC, "outflow": O.TRANSMISSIVE,
         "mixed": (O.PERIODIC, O.PERIODIC, O.TRANSMISSIVE, O.TRANSMISSIVE),
         "walls": (O.REFLECTIVE, O.TRANSMISSIVE, O.REFLECTIVE, O.REFLECTIVE)}


@pytest.mark.parametrize("system", SYSTEMS)
@pytest.mark.parametrize("k,basis", KB)
def test_zeros_stay_exactly_zero(k, basis, system):
    """A state of zeros (either sign), and an Euler state without momentum: its
    right-hand side, damping and sigma are zeros, not the last unit of a block (a
    field that is 0 everywhere takes no part in delta)."""
    p, ctx = _pair(system, k, basis, 11, 6, by=0.5)
    u = _state(p, np.random.default_rng(k))
    if system == O.EULER:
        u[:, 1:3] = 0.0
        zero = [1, 2]
    else:
        u[:] = 0.0
        zero = [0]
    u[:, zero, ::2] = -0.0
    ug = torch.from_numpy(u).cuda()
    d = torch.zeros((2, p.ny, p.nx, p.k + 1), dtype=torch.float64, device="cuda")
    s = torch.zeros((2, p.nfields), dtype=torch.float64, device="cuda")
    ctx.cdg_oe_coefficients(ug, d, s)
    ref, _, _, st = O.oe_coefficients(p, u)
    assert st == O.OK and (s.cpu().numpy()[:, zero] == 0.0).all()
    # differences and sigma of 0.02 from averages of 4: 100 roundings of 2^-53 x 200
    assert np.abs(d.cpu().numpy() - ref).max() <= 3e-12 * np.abs(ref).max()
    L, out = torch.ones_like(ug), torch.ones_like(ug)
    ctx.cdg_rhs(ug, 1e-3, L)
    ctx.cdg_set_dt(1e-3, 1e-3)
    ctx.cdg_oe_damp(ug, out)
    assert (out[:, zero] == 0.0).all()
    if system != O.EULER:
        assert (L == 0.0).all()
        ctx.cdg_rk_stage(0, ug, ug, out)
        assert (out == 0.0).all()


def test_a_transverse_momentum_of_zero_stays_zero():
    """Q^2 Euler, data that vary along one axis only and have no momentum across it:
    the fluxes of that momentum are the pressure, whose differences cancel exactly in
    every mode but those of the faces' sums."""
    for axis in (1, 2):  # the field without momentum: x, y
        p, ctx = _pair(O.EULER, 2, O.BASIS_Q, 10, 9)
        rng = np.random.default_rng(axis)
        u = _state(p, rng, 0.05)
        u[:, axis] = 0.0
        for m, (a, b) in enumerate(p.modes()):
            if (a if axis == 1 else b) > 0:
                u[:, :, m] = 0.0
        u[:] = u[:, :, :, :, :1] if axis == 1 else u[:, :, :, :1, :]
        L = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
        ctx.cdg_rhs(torch.from_numpy(u).cuda(), 1e-3, L)
        L = L.cpu().numpy()
        for m, (a, b) in enumerate(p.modes()):
            if (a if axis == 1 else b) == 0:
                assert (L[:, axis, m] == 0.0).all(), (axis, m)


@pytest.mark.parametrize("nx,ny,by", [(13, 6, 0.7), (9, 7, 3.0), (17, 3, 1.0)])
@pytest.mark.parametrize("sides", sorted(SIDES))
@pytest.mark.parametrize("system", SYSTEMS)
@pytest.mark.parametrize("k,basis", KB)
def test_a_stage_is_the_combination_of_its_right_hand_side(k, basis, system, sides, nx, ny, by):
    """The fused stage of every (system, sides, space) against 3/4 u^n + 1/4 (u_l +
    tau L) formed from cdg_rhs, on ragged meshes of oblong cells.  Both round some
    tens of terms of at most |u| at 2^-53: 1e-14 of max |u|."""
    if sides == "walls" and system != O.EULER:
        pytest.skip("walls need the Euler equations")
    p, ctx = _pair(system, k, basis, nx, ny, by=by, bc=SIDES[sides])
    rng = np.random.default_rng(nx)
    un, ul = (torch.from_numpy(_state(p, rng)).cuda() for _ in range(2))
    L, out = torch.zeros_like(ul), torch.zeros_like(ul)
    tau, tm = 0.6e-3, 0.8e-3
    ctx.cdg_rhs(ul, tm, L)
    ctx.cdg_set_dt(tau, tm)
    ctx.cdg_rk_stage(1, un, ul, out)
    ref = 0.75 * un + 0.25 * (ul + tau * L)
    assert float((out - ref).abs().max()) <= 1e-14 * float(ul.abs().max())


@pytest.mark.parametrize("basis", [O.BASIS_Q, O.BASIS_P])
def test_more_rows_than_a_grid_dimension_of_tiles(basis):
    """131080 rows in tiles of 2 at k = 3: data of period 8 in y give the rows of the
    8-row mesh, bit for bit (the cells are alike: h = 1 on both)."""
    reps = 16385
    p, small = _pair(O.ADVECTION, 3, basis, 3, 8, bx=3.0, by=8.0)
    _, tall = _pair(O.ADVECTION, 3, basis, 3, 8 * reps, bx=3.0, by=8.0 * reps)
    u = torch.from_numpy(_state(p, np.random.default_rng(1))).cuda()
    v = u.repeat(1, 1, 1, reps, 1).contiguous()
    a, b = torch.zeros_like(u), torch.zeros_like(v)
    small.cdg_rhs(u, 1e-2, a)
    tall.cdg_rhs(v, 1e-2, b)
    assert torch.equal(b, a.repeat(1, 1, 1, reps, 1))
    for ctx, x, out in ((small, u, a), (tall, v, b)):
        ctx.cdg_set_dt(0.5e-2, 1e-2)
        ctx.cdg_rk_stage(0, x, x, out)
    assert torch.equal(b, a.repeat(1, 1, 1, reps, 1))
    d, s = torch.zeros((2, 8 * reps, 3, 4), dtype=torch.float64, device="cuda"), torch.zeros((2, 1), dtype=torch.float64, device="cuda")
    tall.cdg_oe_coefficients(v, d, s)
    assert torch.equal(d, d[:, :8].repeat(1, reps, 1, 1)) and float(d.min()) > 0.0


def _delta(ctx, p, u):
    d = torch.zeros((2, p.ny, p.nx, p.k + 1), dtype=torch.float64, device="cuda")
    ctx.cdg_oe_coefficients(torch.from_numpy(u).cuda(), d, None)
    return d.cpu().numpy()


@pytest.mark.parametrize("along", [0, 1])
@pytest.mark.parametrize("aspect", [10.0, 100.0, 1e4])
@pytest.mark.parametrize("k,basis", KB)
def test_coefficients_of_oblong_cells(k, basis, aspect, along):
    """Data that vary along the longer side only: every cell's delta^m, whose derivatives
    the m-th power of the aspect ratio scales down, to the rounding of some tens of terms
    (a sum of norms, so nothing cancels behind the point values: 1e-12)."""
    n, h = (8, 6), ((aspect, 1.0) if along == 0 else (1.0, aspect))
    p, ctx = _pair(O.ADVECTION, k, basis, *n, bx=n[0] * h[0], by=n[1] * h[1])
    u = np.random.default_rng(k).standard_normal(p.shape)
    for m, ab in enumerate(p.modes()):
        if ab[1 - along]:
            u[:, :, m] = 0.0
    u[:] = u[:, :, :, :1, :] if along == 0 else u[:, :, :, :, :1]
    ref, _, _, st = O.oe_coefficients(p, u)
    assert st == O.OK and ref.min() > 0.0
    assert (np.abs(_delta(ctx, p, u) - ref) / ref).max() <= 1e-12


@pytest.mark.parametrize("system", SYSTEMS)
@pytest.mark.parametrize("k,basis", KB)
def test_coefficients_far_below_the_variation(k, basis, system):
    """Modes that fall off as 2^-8 per degree, as resolved data's: delta^k is taken from
    the highest ones, exactly, whatever the size of the lower ones (1e-12 as above)."""
    p, ctx = _pair(system, k, basis, 11, 6, by=0.5)
    rng = np.random.default_rng(k)
    u = _state(p, rng, 0.0)
    for m, (a, b) in enumerate(p.modes()):
        u[:, :, m] += 2.0 ** (-4 - 8 * (a + b)) * rng.uniform(0.5, 1.0, u[:, :, m].shape) * rng.choice([-1.0, 1.0], u[:, :, m].shape)
    ref, _, _, st = O.oe_coefficients(p, u)
    assert st == O.OK
    assert (np.abs(_delta(ctx, p, u) - ref)[..., k] / ref[..., k]).max() <= 1e-12


@pytest.mark.parametrize("along", [0, 1])
@pytest.mark.parametrize("aspect", [8.0, 64.0, 1e4])
@pytest.mark.parametrize("k,basis", KB)
def test_damping_of_oblong_cells(k, basis, aspect, along):
    """Averages that vary along the longer side, modes of degree 1 and more along the
    shorter one by 2^-s smaller (s = 0..40: from complete decay to none), h_min = 1, tau =
    0.1: a decay's argument rounds some 50 times, 0.37 x 50 x 2^-53 of the largest mode."""
    n, h = (8, 6), ((aspect, 1.0) if along == 0 else (1.0, aspect))
    p, ctx = _pair(O.ADVECTION, k, basis, *n, bx=n[0] * h[0], by=n[1] * h[1])
    ctx.cdg_set_dt(0.1, 0.1)
    for s in range(0, 44, 4):
        rng = np.random.default_rng(s)
        u = rng.standard_normal(p.shape)
        u[:, :, 0] = u[:, :, 0, :1, :] if along == 0 else u[:, :, 0, :, :1]
        for m, ab in enumerate(p.modes()):
            if ab[1 - along]:
                u[:, :, m] *= 2.0 ** -s
        ug = torch.from_numpy(u).cuda()
        out = torch.zeros_like(ug)
        ctx.cdg_oe_damp(ug, out)
        ref, st = O.oe(p, u, 0.1)
        assert st == O.OK
        assert np.abs(out.cpu().numpy() - ref).max() <= 2e-15 * np.abs(u).max(), s


@pytest.mark.parametrize("power", [1018, -930])
@pytest.mark.parametrize("k,basis", KB)
def test_linear_results_scale_with_the_data(k, basis, power):
    """Advection of data times a power of two, up to the last ones whose sums are finite:
    right-hand side, stage and damping are the unscaled ones times it, bit for bit (2 x 2
    cells, so that the sum of the averages is finite too)."""
    p, ctx = _pair(O.ADVECTION, k, basis, 2, 2)
    u = torch.from_numpy(0.5 * _state(p, np.random.default_rng(k), 0.05)).cuda()
    tau, tm = 2.0 ** -9, 2.0 ** -8
    ctx.cdg_set_dt(tau, tm)
    s, got = 2.0 ** power, []
    for x in (u, u * s):
        L, stage, damped = torch.zeros_like(u), torch.zeros_like(u), torch.zeros_like(u)
        ctx.cdg_rhs(x, 1.0, L)
        ctx.cdg_rk_stage(0, x, x, stage)
        ctx.cdg_oe_damp(x, damped)
        got.append((L, stage, damped))
    for a, b in zip(*got):
        assert torch.isfinite(b).all() and torch.equal(a * s, b)


@pytest.mark.parametrize("system", SYSTEMS)
@pytest.mark.parametrize("k,basis", KB)
def test_infinities_and_nans_give_nan(k, basis, system):
    """One value that is not finite makes the right-hand side NaN in the cells that
    overlap it, and no other."""
    for bad in (float("inf"), float("-inf"), float("nan")):
        p, ctx = _pair(system, k, basis, 12, 7)
        u = _state(p, np.random.default_rng(k))
        u[0, 0, 0, 3, 5] = bad
        L = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
        ctx.cdg_rhs(torch.from_numpy(u).cuda(), 1e-3, L)
        L = L.cpu().numpy()
        finite = np.isfinite(L).all(axis=(1, 2))
        near = np.zeros(finite.shape, bool)
        near[1, 2:4, 4:6] = True  # dual cells over primal (5, 3)
        near[0, 3, 5] = True  # its own -u / tau term
        assert (finite == ~near).all()
        assert np.isnan(L[1, 0, 0, 2:4, 4:6]).all()


@pytest.mark.parametrize("system", SYSTEMS)
@pytest.mark.parametrize("k,basis", KB)
def test_a_nan_mode_leaves_sigma_to_the_other_cells(k, basis, system):
    """One cell's highest mode is NaN beside the cells that hold the extrema of their
    fields: that mesh's sigma is the one without the cell's variation."""
    p, ctx = _pair(system, k, basis, 12, 7)
    u = _state(p, np.random.default_rng(k))
    u[0, :, 0, 0, 0] += 0.3  # the extremum, in the same tile
    u[0, :, 1:, 0, 3] = 0.0
    v = u.copy()
    v[0, :, -1, 0, 3] = np.nan
    s, t = (torch.zeros((2, p.nfields), dtype=torch.float64, device="cuda") for _ in range(2))
    ctx.cdg_oe_coefficients(torch.from_numpy(u).cuda(), None, s)
    ctx.cdg_oe_coefficients(torch.from_numpy(v).cuda(), None, t)
    assert float(s.min()) > 0.0 and torch.equal(s[0], t[0])


@pytest.mark.parametrize("gamma", [1.0 + 2.0 ** -10, 1.4, 3.0])
@pytest.mark.parametrize("low", [0.5, 2.0 ** -4, 2.0 ** -6, 2.0 ** -7, 2.0 ** -10, -(2.0 ** -10), -0.25])
def test_fluxes_at_densities_close_to_zero(low, gamma):
    """Q^2 Euler: cells whose density falls to `low` at one Gauss point, at every place of an
    8-cell warp and in the ragged tile.  The largest flux of such a quarter is far below the
    product of its factors' exponents, so its warp takes the fluxes in FP64; on either
    side of that line.  A density rounds at about 2^-53 x 8 there and its flux by twice
    the quotient: 2e-15 / |low|, and some tens of roundings in the sums: 1e-13 / min(1,
    |low|) of a field's largest right-hand side."""
    p, ctx = _pair(O.EULER, 2, O.BASIS_Q, 11, 6, bx=11 / 8, by=6 / 8, gamma=gamma)
    u = _state(p, np.random.default_rng(3))
    x = 0.5 + 0.5 * 0.6 ** 0.5  # the quarter's outer Gauss point in the overlapping cell
    for mesh in range(2):
        for n in range(8):
            cell = (3 * n) % p.ny, n if mesh == 0 else n + 3
            u[(mesh, 0, slice(1, None)) + cell] = 0.0
            u[(mesh, 0, 0) + cell] = 1.0
            u[(mesh, 0, 1) + cell] = (-1.0) ** n * (1.0 - low) / x
    L = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    ctx.cdg_rhs(torch.from_numpy(u).cuda(), 1 / 64, L)
    ref = O.rhs(p, u, 1 / 64)
    err = np.abs(L.cpu().numpy() - ref).max(axis=(0, 2, 3, 4)) / np.abs(ref).max(axis=(0, 2, 3, 4))
    assert err.max() <= 1e-13 / min(1.0, abs(low)), err


@pytest.mark.parametrize("gamma", [1.0 + 2.0 ** -10, 1.4, 3.0])
@pytest.mark.parametrize("speed", [0.0, 1e-6, 1e3])
def test_cells_at_rest_and_cold_fast_flow(speed, gamma):
    """Q^2 Euler at Mach numbers from 0 to some thousands: the energy and momentum fluxes
    to 1e-13 of the largest of their equations' terms (flux over h, the state over tau)."""
    p, ctx = _pair(O.EULER, 2, O.BASIS_Q, 11, 6, bx=11 / 8, by=6 / 8, gamma=gamma)
    rng = np.random.default_rng(5)
    u = _state(p, rng)
    u[:, 1:3] = 0.0
    if speed:
        u[:, 1, 0] = speed * (1.0 + 0.01 * rng.standard_normal(u[:, 1, 0].shape))
        u[:, 2, 1:] = 1e-3 * speed * rng.standard_normal(u[:, 2, 1:].shape)
        u[:, 3, 0] += 0.6 * speed ** 2
    L = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    ctx.cdg_rhs(torch.from_numpy(u).cuda(), 1 / 64, L)
    ref = O.rhs(p, u, 1 / 64)
    top = np.abs(u[:, 3]).max()
    scale = np.array([1.0 + speed, top, top, top * (1.0 + speed)]) * 64 * 9
    err = np.abs(L.cpu().numpy() - ref).max(axis=(0, 2, 3, 4)) / scale
    assert err.max() <= 1e-13, err


def test_a_tuning_file_of_other_kernels_is_not_used(tmp_path):
    """An entry without the kernels' generation (as the FP64 kernels wrote it) is kept in
    the file, and the batch is tuned anew."""
    from paper_2503_12473_gb300 import oecdg as G
    descs = [G.MeshDesc(dim=2, nx=nx, ny=ny, system=G.EULER, bc=G.PERIODIC, cfl=0.1) for nx, ny in ((8, 12), (20, 9))]
    h = 1469598103934665603
    for d in descs:
        for n in (d.nx, d.ny):
            h = (h ^ n) * 1099511628211 % 2 ** 64
    old = {f"euler_q2_bc0_n2_{h:016x}": 801}
    path = tmp_path / "tune.json"
    path.write_text(json.dumps(old))
    us = []
    for d in descs:
        p = O.Problem(dim=2, nx=d.nx, ny=d.ny, k=2, system=O.EULER, bc=O.PERIODIC)
        us.append(torch.from_numpy(_state(p, np.random.default_rng(d.nx))).cuda())
    b = G.Batch(descs)
    rows = b.cdg_batch_autotune(us, str(path))
    new = json.loads(path.read_text())
    assert len(new) == 2 and new.pop(next(iter(old))) == 801
    assert list(new.values()) == [100 * rows + b.cdg_batch_grid()[0]]


@pytest.mark.parametrize("bx,by", [(6.0, 1.0), (1.0, 3.0)])
@pytest.mark.parametrize("sides", sorted(SIDES))
@pytest.mark.parametrize("system", [O.EULER, O.ADVECTION])
@pytest.mark.parametrize("k,basis", [(2, O.BASIS_Q), (3, O.BASIS_P)])
def test_steps_on_oblong_cells(k, basis, system, sides, bx, by):
    """Damping and two steps at aspect ratios of 3 to 6 either way, every side
    condition: 1e-12 relative L1, as elsewhere for two steps of smooth data."""
    if sides == "walls" and system != O.EULER:
        pytest.skip("walls need the Euler equations")
    p, ctx = _pair(system, k, basis, 13, 12, bx=bx, by=by, bc=SIDES[sides], rk=k + 1)
    u = _state(p, np.random.default_rng(7))
    ug = torch.from_numpy(u).cuda()
    out = torch.zeros_like(ug)
    ctx.cdg_set_dt(0.7e-3, 1e-3)
    ctx.cdg_oe_damp(ug, out)
    ref, st = O.oe(p, u, 0.7e-3)
    assert st == O.OK and np.abs(out.cpu().numpy() - ref).sum() <= 1e-12 * np.abs(ref).sum()
    ctx.cdg_step(ug, 0.0, 0.0, 2)
    ref, _, n, st = O.advance(p, u, 0.0, 0.0, 2)
    assert st == O.OK and n == 2 and np.abs(ug.cpu().numpy() - ref).sum() <= 1e-12 * np.abs(ref).sum()


@pytest.mark.parametrize("bx,by", [(10.0, 1.0), (1.0, 6.0)])
@pytest.mark.parametrize("system,nx,ny", [(O.ADVECTION, 6, 5), (O.EULER, 4, 3)])
def test_adjoint_on_oblong_cells(system, nx, ny, bx, by):
    """J^T lam of a step with the OE step's recorded sums on cells of aspect ratio 4 to 8
    against the oracle's own adjoint (complex step), with the bars of square cells."""
    p, ctx = _pair(system, 2, O.BASIS_Q, nx, ny, bx=bx, by=by)
    rng = np.random.default_rng(4)
    u = 0.05 * rng.uniform(-1.0, 1.0, p.shape)
    if system == O.EULER:
        u[:, 0, 0] += 1.0
        u[:, 3, 0] += 2.5
    lam = rng.uniform(-1.0, 1.0, p.shape)
    ref, st = O.step_adjoint(p, u, lam)
    assert st == O.OK
    got = torch.empty(p.shape, dtype=torch.float64, device="cuda")
    ctx.cdg_step_adjoint(torch.from_numpy(u).cuda(), torch.from_numpy(lam).cuda(), got)
    err = np.abs(got.cpu().numpy() - ref)
    assert err.sum() <= 1e-10 * np.abs(ref).sum() and err.max() <= 1e-9 * np.abs(ref).max()
