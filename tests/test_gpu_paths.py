"""Kernel paths that a mesh's size, alignment or datum selects, at the sizes where they change.

Tile rows inside the mesh (wider than one 32-cell tile on both sides) against the general copies of
a state that is not 16-byte aligned; the separable Fourier projection and the general one; the
CFL maximum; the positivity limiter inside the stage kernel against its own launch; the troubled
cells of a tile, from none to all; CG node tiles on both sides of their width rule; the totals.
"""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2601_16911_gb300 import cvweno as cv
from paper_2601_16911_gb300 import inputs as I
from tests.gpu_common import ALPHA_TOL, GAMMA_TOL, RES_TOL, rel_err, rounded, to_gpu
from tests.test_gpu_alignment import misaligned_copy
from tests.test_oracle_positivity import random_state

pytestmark = pytest.mark.gpu


ROWS = ([("kpp", p, I.DG) for p in (1, 2, 3, 4)] + [("kpp", p, I.CG) for p in (1, 2, 3, 4)]
        + [("euler", p, I.DG) for p in (1, 2, 3, 4)])


@pytest.mark.parametrize("nx,ny", [(64, 9), (67, 13), (97, 33)])
@pytest.mark.parametrize("system,p,kind", ROWS, ids=["%s-%s-q%d" % (s, "cg" if k else "dg", p) for s, p, k in ROWS])
def test_interior_tiles_agree_with_unaligned_loads(system, p, kind, nx, ny):
    # the copies differ, the arithmetic does not: equal bits
    if system == "kpp":
        d, ic = I.kpp(3, n=nx, degree=p, kind=kind)
        d = dict(d, ny=ny)
    else:
        d, ic = I.euler_quadrants(2, n=nx, degree=p)
        d = dict(d, ny=ny)
    m = cv.Mesh(d)
    u = m.project(*ic)
    ua, um = u.clone(), misaligned_copy(u)
    ra, rm = m.residual(ua), m.residual(um)
    m.advance(ua, 2e-5, 2)
    m.advance(um, 2e-5, 2)
    torch.cuda.synchronize()
    m.status_check()
    assert torch.equal(ra, rm)
    assert torch.equal(ua, um) and not torch.equal(ua, u)
    m.close()


def fourier(modes):
    return [float(len(modes))] + [x for m in modes for x in m]


FOURIER = {
    "none": fourier([]),
    "one": fourier([(1.5, 0.0, 2.0, -0.7)]),
    "negative": fourier([(0.5, -3.0, 1.0, 7.0), (-1.0, 2.0, -5.0, 0.1)]),
    "fifteen": fourier([(0.1 * (k + 1), float(k % 6), float((2 * k) % 5), 0.4 * k) for k in range(15)]),
}


@pytest.mark.parametrize("modes", list(FOURIER))
@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 130), (129, 33)])
def test_fourier_projection(p, nx, ny, modes):
    d = I.mesh(2, nx, ny, degree=p, system=I.BURGERS, domain=(-0.3, 1.1, 2.0, 2.5))
    prm = FOURIER[modes]
    ref = O.project(d, I.IC_FOURIER, prm)
    mesh = cv.Mesh(d)
    u = mesh.project(I.IC_FOURIER, prm)
    um = misaligned_copy(torch.zeros_like(u))
    mesh.project(I.IC_FOURIER, prm, out=um)
    got = u.cpu().numpy()
    assert torch.equal(u, um)
    mesh.close()
    # a mode is a sum of two products of an x and a y factor; each factor is a rotation of two
    # FP32 numbers and the phase another: about 8 roundings on |a| times the factors' size, at
    # most 4 for the Legendre projections met here
    bound = 32 * 2.0 ** -24 * sum(abs(a) for a in prm[1::4])
    assert np.abs(got - ref).max() <= bound, (np.abs(got - ref).max(), bound)


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("dim,nx,ny", [(1, 1, 1), (1, 130, 1), (2, 1, 1), (2, 3, 51), (2, 65, 17)])
def test_general_projection(p, dim, nx, ny):
    d = I.mesh(dim, nx, ny, degree=p, system=I.BURGERS)
    data = [(I.IC_POLY, [0.3 * ((i * 7) % 5) - 0.6 for i in range(25)])]
    if dim == 1:
        data.append((I.IC_FOURIER, fourier([(1.0, 2.0, 0.0, 0.3), (0.5, -1.0, 0.0, 1.0)])))
    else:
        data.append((I.IC_CIRCLE, [0.4, 0.6, 0.27, 2.0, -1.0]))
    mesh = cv.Mesh(d)
    for ic in data:
        # the 12-point rule in FP32: a few ulps of the largest coefficient
        assert rel_err(mesh.project(*ic).cpu().numpy(), O.project(d, *ic)) < 2e-6
    mesh.close()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("system,dim,nx,ny", [(I.BURGERS, 1, 1, 1), (I.BURGERS, 1, 1031, 1), (I.LINADV, 2, 7, 3),
                                              (I.BURGERS, 2, 1, 1), (I.KPP, 2, 33, 129), (I.BURGERS, 2, 301, 150),
                                              (I.EULER, 2, 1, 1), (I.EULER, 2, 19, 11), (I.EULER, 2, 130, 67)])
def test_max_wavespeed(system, dim, nx, ny, p):
    d = I.mesh(dim, nx, ny, degree=p, system=system)
    rng = np.random.default_rng(p + nx)
    u = random_state(d, rng, 0.05) if system == I.EULER else rng.standard_normal(O.state_shape(d)) * 0.5
    u = rounded(u)
    ref = O.max_wavespeed(d, u)
    mesh = cv.Mesh(d)
    big, small = to_gpu(u), to_gpu(u) if system == I.EULER else to_gpu(0.25 * u)
    first = mesh.max_wavespeed(big)
    mesh.max_wavespeed(small)
    assert mesh.max_wavespeed(misaligned_copy(big)) == first  # nothing is left of an earlier call
    assert abs(first - ref) <= 1e-6 * ref
    mesh.close()


@pytest.mark.parametrize("kind", [I.DG, I.CG], ids=["dg", "cg"])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_an_infinite_state_has_no_finite_speed(kind, p):
    d = I.mesh(2, 40, 13, degree=p, system=I.BURGERS, kind=kind)
    mesh = cv.Mesh(d)
    u = 0.02 * torch.sin(torch.arange(mesh.empty_state().numel(), device="cuda", dtype=torch.float32)).view_as(mesh.empty_state())
    u.view(-1)[7 * u.shape[-1] % u.numel()] = float("inf")  # a DG cell's mean; a CG node
    assert mesh.max_wavespeed(u) == float("inf")
    mesh.close()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("nx,ny", [(19, 11), (67, 21)])
def test_positivity_in_the_stage_matches_its_own_launch(p, nx, ny):
    d = I.mesh(2, nx, ny, degree=p, system=I.EULER, bc=I.TRANSMISSIVE, positivity=1)
    u0 = to_gpu(random_state(d, np.random.default_rng(20 + p), 0.25))
    a, b = cv.Mesh(d), cv.Mesh(d)
    b.set_kernel_timing(True)  # the limiter as a launch of its own
    a.positivity(u0, out=u0)
    ua, ub = u0.clone(), u0.clone()
    dt = 0.02 / (max(nx, ny) * 4.0 * (2 * p + 1))
    a.advance(ua, dt, 1)
    b.advance(ub, dt, 1)
    torch.cuda.synchronize()
    assert len(b.kernel_times()) == 6
    a.status_check()
    b.status_check()
    # the same limiter on the same stage results: the bar of the limiter itself
    assert rel_err(ua.cpu().numpy().astype(np.float64), ub.cpu().numpy().astype(np.float64)) <= 1e-5
    a.close()
    b.close()


TROUBLED = [(I.DG, 1, I.BURGERS, 131, 1), (I.DG, 2, I.KPP, 35, 9), (I.CG, 2, I.KPP, 19, 9), (I.CG, 1, I.BURGERS, 131, 1)]


@pytest.mark.parametrize("share", [0.0, 0.02, 1.0])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("kind,dim,system,nx,ny", TROUBLED, ids=["dg1d", "dg2d", "cg2d", "cg1d"])
def test_troubled_share(kind, dim, system, nx, ny, p, share):
    d = I.mesh(dim, nx, ny, degree=p, system=system, kind=kind)
    rng = np.random.default_rng(p)
    u = rounded(rng.standard_normal(O.state_shape(d)) * 0.5)
    ov = (rng.uniform(size=O.counts(d)["ncell"]) < share).astype(np.int32)
    ref = O.residual(d, u, ov)
    mesh = cv.Mesh(d)
    out = mesh.residual_ex(to_gpu(u), troubled_override=torch.from_numpy(ov).cuda())
    mesh.status_check()
    got = {k: v.cpu().numpy() for k, v in out.items()}
    mesh.close()
    assert np.array_equal(got["troubled"], ref["troubled"])
    assert np.abs(got["alpha"] - ref["alpha"]).max() <= ALPHA_TOL * np.abs(ref["alpha"]).max()
    assert rel_err(got["dudt"], ref["dudt"]) < RES_TOL


@pytest.mark.parametrize("p", [3, 4])
def test_cg_node_tiles_of_both_widths(p):
    # A small periodic mesh and the same state repeated 4 x 4 times on four times the domain: the
    # residual of every copy is the small mesh's, whose lattice takes the narrow node tiles.
    n = 60 if p == 3 else 47
    d = I.mesh(2, n, n - 1, degree=p, system=I.BURGERS, kind=I.CG)
    big = dict(d, nx=4 * d["nx"], ny=4 * d["ny"], x1=4.0, y1=4.0)
    m, mb = cv.Mesh(d), cv.Mesh(big)
    u = m.project(I.IC_FOURIER, FOURIER["fifteen"])
    ub = u.view(p * d["ny"], p * d["nx"]).repeat(4, 4).contiguous().view(mb.empty_state().shape)
    r = m.residual(u).view(p * d["ny"], p * d["nx"]).repeat(4, 4)
    rb = mb.residual(ub).view(4 * p * d["ny"], 4 * p * d["nx"])
    m.status_check()
    mb.status_check()
    assert (r - rb).abs().max().item() <= RES_TOL * r.abs().max().item()
    m.close()
    mb.close()


@pytest.mark.parametrize("system,nx,ny,p", [(I.BURGERS, 1, 1, 1), (I.KPP, 257, 3, 2), (I.EULER, 130, 67, 3)])
def test_totals(system, nx, ny, p):
    d = I.mesh(2, nx, ny, degree=p, system=system)
    u = rounded(np.random.default_rng(nx).standard_normal(O.state_shape(d)))
    mesh = cv.Mesh(d)
    ug = to_gpu(u)
    got = [mesh.mass_total(ug) for _ in range(3)]
    ref = O.mass_total(d, u)
    assert got[0] == got[1] == got[2]
    # FP64 sums of the same numbers in another order
    assert np.abs(np.array(got[0]) - np.asarray(ref)).max() <= 1e-12 * np.abs(u[:, :, 0]).sum()
    mesh.close()


@pytest.mark.parametrize("p", [1, 2, 4])
def test_a_wave_speed_call_counts_its_fallbacks(p):
    # conf_min = 1: every cell that is not flat falls back in every evaluation of the sensor, the one of
    # a wave-speed call among them: a CFL-controlled step counts four times what a residual does
    d = I.mesh(2, 21, 17, degree=p, system=I.BURGERS)
    rng = np.random.default_rng(p)
    u = to_gpu(rounded(rng.standard_normal(O.state_shape(d)) * 0.5))
    net = cv.Mlp(np.array(I.mlp_init(5)))
    mesh = cv.Mesh(d)
    plain = mesh.max_wavespeed(u)
    mesh.set_surrogate(net, conf_min=1.0)
    mesh.residual(u)
    once = net.fallbacks(reset=True)
    assert once == d["nx"] * d["ny"]
    speed = mesh.max_wavespeed(u)
    assert net.fallbacks(reset=True) == once
    assert abs(speed - plain) <= 1e-6 * plain
    mesh.step(u, cfl=0.01)
    assert net.fallbacks(reset=True) == 4 * once
    mesh.set_surrogate(None)
    mesh.close()
    net.close()


@pytest.mark.parametrize("direction", [0, 1])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_euler_wave_speed_keeps_modes_below_an_ulp_of_the_mean(p, direction):
    # p modes of 0.49 ulp of the mean each: their sum at one side of the cell is added to the mean
    # there, so the speed is, to the bit, that of a cell whose mean has the rounded sum
    d = I.mesh(2, 5, 3, degree=p, system=I.EULER, bc=I.TRANSMISSIVE)
    n, mesh = p + 1, cv.Mesh(d)
    rho, E = np.float32(1.0 + 8 * 2.0 ** -23), np.float32(2.0 + 8 * 2.0 ** -22)
    base = np.zeros(O.state_shape(d), np.float32)
    base[0, :, 0], base[3, :, 0] = rho, E
    modes, whole = base.copy(), base.copy()
    for v, mean, sign in ((0, rho, -1.0), (3, E, 1.0)):  # less dense and hotter: faster
        part = np.float32(sign * 0.49 * np.spacing(mean))
        for m in range(1, n):
            modes[v, 7, m if direction == 0 else n * m] = part
        whole[v, 7, 0] = np.float32(np.float64(mean) + p * np.float64(part))
    still, got, want = (mesh.max_wavespeed(to_gpu(u)) for u in (base, modes, whole))
    assert want > still
    assert got == want
    mesh.close()


def limited_step(d, u, dt, without=None):
    """One limited SSP-RK3 step by the oracle (the limiter left out after stage `without`) and the
    number of cells limited after each stage."""
    plain, w, limited = dict(d, positivity=0), u, []
    for k, (a, b) in enumerate(((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))):
        w = a * u + b * (w + dt * O.residual(plain, w)["dudt"].reshape(w.shape))
        if k != without:
            w, theta, _ = O.positivity(d, w)
            limited.append(int((theta < 1.0).sum()))
    return w, limited


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("nx,ny,seed", [(35, 19, 0), (20, 33, 1)])
def test_positivity_in_the_stage_limits_in_every_stage(p, nx, ny, seed):
    # pressures at the limiter's floor in many cells of several tiles: it acts after all three stages
    d = I.mesh(2, nx, ny, degree=p, system=I.EULER, bc=I.TRANSMISSIVE, positivity=1)
    u0 = rounded(O.positivity(d, random_state(d, np.random.default_rng(20 + p + seed), 1.6))[0])
    dt = 0.2 / (max(nx, ny) * O.max_wavespeed(d, u0) * (2 * p + 1) * p)
    ref, limited = limited_step(d, u0, dt)
    assert min(limited) > 10
    norm = np.abs(ref).max()
    # near vacuum the step amplifies rounding: the bar is 32 times what one FP32 rounding of every input
    # coefficient does to the FP64 step (some ten roundings of that size in each of three stages)
    sens = 2.0 ** -23
    for s in range(2):
        noise = np.random.default_rng(s).uniform(-1.0, 1.0, u0.shape)
        sens = max(sens, np.abs(limited_step(d, u0 * (1.0 + 2.0 ** -23 * noise), dt)[0] - ref).max() / norm)
    tol = 32.0 * sens
    assert np.abs(limited_step(d, u0, dt, without=2)[0] - ref).max() > 8.0 * tol * norm  # a lost limiter shows
    fused, own = cv.Mesh(d), cv.Mesh(d)
    own.set_kernel_timing(True)  # the limiter as a launch of its own
    got = []
    for m in (fused, own):
        u = to_gpu(u0)
        m.advance(u, dt, 1)
        m.status_check()
        got.append(u.cpu().numpy().astype(np.float64).reshape(u0.shape))
    assert len(own.kernel_times()) == 6
    fused.close()
    own.close()
    assert np.abs(got[0] - ref).max() <= tol * norm
    assert np.abs(got[1] - ref).max() <= tol * norm
    assert np.abs(got[0] - got[1]).max() <= tol * norm


def test_cg_q2_cell_kernels_on_both_sides_of_one_block_per_sm():
    # as the node tiles above: 15 blocks, and 200 for the same state repeated 4 x 4 times
    d = I.mesh(2, 40, 39, degree=2, system=I.BURGERS, kind=I.CG)
    big = dict(d, nx=160, ny=156, x1=4.0, y1=4.0)
    m, mb = cv.Mesh(d), cv.Mesh(big)
    u = m.project(I.IC_FOURIER, FOURIER["fifteen"])
    ub = u.view(78, 80).repeat(4, 4).contiguous().view(mb.empty_state().shape)
    ov = torch.from_numpy((np.random.default_rng(2).uniform(size=(39, 40)) < 0.1).astype(np.int32)).cuda()
    out = m.residual_ex(u, troubled_override=ov.view(-1))
    outb = mb.residual_ex(ub, troubled_override=ov.repeat(4, 4).contiguous().view(-1))
    m.status_check()
    mb.status_check()
    r, rb = out["dudt"].view(78, 80).repeat(4, 4), outb["dudt"].view(312, 320)
    assert (r - rb).abs().max().item() <= RES_TOL * r.abs().max().item()
    g, gb = out["gamma"].view(39, 40).repeat(4, 4), outb["gamma"].view(156, 160)
    assert (g - gb).abs().max().item() <= GAMMA_TOL
    m.close()
    mb.close()


@pytest.mark.parametrize("nx,ny", [(192, 96), (208, 104)])  # 144 and 169 blocks
@pytest.mark.parametrize("system", [I.BURGERS, I.KPP, I.LINADV])
def test_cg_q2_cell_kernels_against_the_oracle(system, nx, ny):
    d = I.mesh(2, nx, ny, degree=2, system=system, kind=I.CG)
    rng = np.random.default_rng(nx)
    u = rounded(rng.standard_normal(O.state_shape(d)) * 0.5)
    ov = (rng.uniform(size=O.counts(d)["ncell"]) < 0.1).astype(np.int32)
    ref = O.residual(d, u, ov)
    mesh = cv.Mesh(d)
    out = mesh.residual_ex(to_gpu(u), troubled_override=torch.from_numpy(ov).cuda())
    mesh.status_check()
    got = {k: v.cpu().numpy() for k, v in out.items()}
    mesh.close()
    assert np.array_equal(got["troubled"], ref["troubled"])
    assert np.abs(got["alpha"] - ref["alpha"]).max() <= ALPHA_TOL * np.abs(ref["alpha"]).max()
    assert rel_err(got["dudt"], ref["dudt"]) < RES_TOL


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("p", [2, 4])
def test_cg_cells_odd_about_their_middle_have_no_even_modes(p, dim):
    # Nodal values c - d_g, ..., c, ..., c + d_g in x with arbitrary d_g, six cells rising and six falling: the
    # even modes beyond the mean are zero, and sums of mirrored nodes about the middle one exactly so.
    # The vertex candidates' highest x-derivative has the highest mode alone.
    n = 12
    d = I.mesh(dim, n, 5 if dim == 2 else 1, degree=p, system=I.BURGERS, kind=I.CG)
    off = np.sort(np.random.default_rng(p).uniform(0.05, 0.4, p // 2))
    off = np.round(off * 2.0 ** 20) / 2.0 ** 20  # every value below is an FP32 number
    shape = np.concatenate([-off[::-1], [0.0], off])
    middles = 1.0 + off[-1] * np.array([1, 3, 5, 7, 9, 11, 11, 9, 7, 5, 3, 1])
    line = np.concatenate([(c + (shape if k < 6 else -shape))[:-1] for k, c in enumerate(middles)])
    assert np.array_equal(line, line.astype(np.float32))
    u = np.tile(line, (p * d["ny"] if dim == 2 else 1, 1))
    mesh = cv.Mesh(d)
    t = mesh.vertex_data(to_gpu(u.reshape(O.state_shape(d))))
    mesh.status_check()
    assert t[:, p].abs().max().item() == 0.0
    assert t[:, 1].abs().max().item() > 1.0
    mesh.close()
