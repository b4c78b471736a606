"""Kernel paths chosen by size, layout or value, at the edges where the choice
changes: raw populations against plain FP64 formulas or against the general
path of the same call."""
import numpy as np
import pytest
import torch

from paper_2512_12213_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

E = {9: np.array([(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]),
     19: np.array([(0, 0, 0)] + [tuple(s * c for c in v) for v in
                                 [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1),
                                  (0, 1, -1)] for s in (1, -1)])}
W = {9: np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4), 19: np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)}
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}


def raw(sim, buf=None):
    """The stored post-collision populations, (Q, nz, ny, nxp), physical units."""
    if buf is None:
        buf = torch.empty(sim.sizes[lbm.BUF_POP_A], dtype=torch.uint8, device="cuda")
        lbm.lbm_save_state(sim.ctx, buf, sim.stream)
    nz, ny, nx = sim.shape
    nxp = (nx + 63) // 64 * 64
    t = DTYPE[{0: "f64", 1: "f32", 2: "f16s", 3: "bf16s"}[sim.cfg.storage]]
    n = sim.Q * nz * ny * nxp
    return buf.view(t)[:n].view(sim.Q, nz, ny, nxp)


# FP32 deviations of the equilibrium: rounded once from 48-bit sums, whose
# error is 2^-46 of the largest term (w max(|rho - 1|, 3 |u|)); nodes whose
# fields are zero, tiny (below the 48-bit split's range) or large take FP64
@pytest.mark.parametrize("stokes", [0, 1])
@pytest.mark.parametrize("box,scale", [((7, 5, 1), 1.0), ((66, 3, 4), 1.0), ((66, 3, 4), 1e-9), ((5, 3, 2), 1e-30)])
def test_equilibrium_from_fields(box, scale, stokes):
    nx, ny, nz = box
    Q = 9 if nz == 1 else 19
    g = np.random.default_rng(3)
    rho = 1.0 + 0.03 * scale * g.uniform(-1, 1, (nz, ny, nx))
    u = 0.08 * scale * g.uniform(-1, 1, (3, nz, ny, nx))
    rho[0, 0, 1], u[:, 0, 0, 1] = 1.0, 0.0                   # at rest
    u[:, 0, 0, 2] = (1e-40, -0.0, 0.0)
    if nz == 1:
        u[2] = 0.0
    sim = lbm.Sim(dict(lattice=Q, nx=nx, ny=ny, nz=nz, tau=0.8, force_model="e", storage="f32", stokes=stokes),
                  inputs.empty_mask(nx, ny, nz), stage=False)
    sim.init_equilibrium(torch.from_numpy(rho).cuda(), torch.from_numpy(u).cuda())
    P = raw(sim)[..., :nx].double().cpu().numpy()
    eu = np.tensordot(E[Q], u, 1)
    quad = 0.0 if stokes else 4.5 * eu * eu - 1.5 * (u * u).sum(0)
    d = W[Q][:, None, None, None] * ((rho - 1.0) + rho * (3 * eu + quad))
    size = W[Q][:, None, None, None] * np.maximum(np.abs(rho - 1.0), 3 * np.abs(u).max(0))
    for a in range(Q):                                       # P_a(x) = f_a(x + E_a)
        moved = lambda t: np.roll(t, tuple(-E[Q][a][::-1]), axis=(0, 1, 2))  # noqa: E731
        bound = 2.0 ** -24 * np.abs(moved(d[a])) + 2.0 ** -44 * moved(size[a]) + 1e-45
        assert np.all(np.abs(P[a] - moved(d[a])) <= bound), a
    f32 = sim.export_f(torch.float32).double().cpu().numpy()
    f64 = sim.export_f(torch.float64).cpu().numpy()          # the stored value plus w in FP64
    assert np.all(np.abs(f32 - f64) <= 2.0 ** -24 * np.abs(f64) * (1 + 2.0 ** -20))
    sim.import_f(torch.from_numpy(f64.astype(np.float32)).cuda())
    back = raw(sim)[..., :nx].double().cpu().numpy()
    for a in range(Q):
        ref = np.roll(f64[a].astype(np.float32).astype(np.float64) - W[Q][a], tuple(-E[Q][a][::-1]), axis=(0, 1, 2))
        assert np.all(np.abs(back[a] - ref) <= 2.0 ** -24 * np.abs(ref) + 2.0 ** -48)
    sim.close()


# infinities and NaN pass through import and export unchanged in kind
@pytest.mark.parametrize("storage", ["f32", "bf16s", "f64"])
def test_non_finite_populations_pass(storage):
    nx, ny, nz = 9, 4, 3
    sim = lbm.Sim(dict(lattice=19, nx=nx, ny=ny, nz=nz, tau=0.8, force_model="e", storage=storage),
                  inputs.empty_mask(nx, ny, nz), stage=False)
    f = torch.full((19, nz, ny, nx), 0.05, dtype=torch.float64, device="cuda")
    f[3, 1, 2, 4], f[7, 0, 0, 0], f[18, 2, 3, 8] = float("inf"), float("-inf"), float("nan")
    for dtype in (torch.float32, torch.float64):
        sim.import_f(f.to(dtype))
        for out in (torch.float32, torch.float64):
            g = sim.export_f(out).double()
            assert torch.equal(torch.isnan(g), torch.isnan(f)) and torch.equal(torch.isinf(g), torch.isinf(f))
            assert torch.equal(g[torch.isinf(f)], f[torch.isinf(f)])
    sim.close()


# the FP64 step scales exactly with the density unit except for 1/rho, whose
# iteration serves 2^-111 .. 2^112 and the plain quotient the rest: an ulp or
# two per step
@pytest.mark.parametrize("exponent", [-130, 40, 130])
@pytest.mark.parametrize("box", [(5, 3, 1), (70, 9, 1), (33, 6, 5)])
def test_fp64_step_density_unit(box, exponent):
    nx, ny, nz = box
    Q = 9 if nz == 1 else 19
    mask = inputs.random_solids(nx, ny, nz, 0.08, seed=2)
    rho, u = inputs.smooth_fields(nx, ny, nz, dims=2 if nz == 1 else 3, u_amplitude=0.04, seed=5)
    out = []
    for r in (1.0, 2.0 ** exponent):
        sim = lbm.Sim(dict(lattice=Q, nx=nx, ny=ny, nz=nz, periodic=(1, 0, 1), tau=0.7, rho0=r, force_model="c",
                           g=(1e-4, -2e-5, 0), storage="f64", wall_u=((0.01, 0, 0),)), mask, stage=False)
        sim.init_equilibrium(torch.from_numpy(rho * r).cuda(), torch.from_numpy(u).cuda())
        sim.step(6)
        out.append(sim.export_f() / r)
        sim.close()
    assert (out[0] - out[1]).abs().max() <= 1e-13 * out[0].abs().max()


# a step into a buffer that is not the context's own zeroes its padding
@pytest.mark.parametrize("storage,kernel", [("f64", "auto"), ("f32", "register"), ("f32", "staged"), ("bf16s", "staged")])
@pytest.mark.parametrize("nx", [41, 66, 130])
def test_step_from_leaves_no_padding(nx, storage, kernel):
    ny, nz = 7, 5
    mask = inputs.random_solids(nx, ny, nz, 0.02, seed=9)
    sim = lbm.Sim(dict(lattice=19, nx=nx, ny=ny, nz=nz, tau=0.7, force_model="e", g=(1e-5, 0, 0), storage=storage,
                       wall_u=((0, 0, 0),), step_kernel=kernel), mask, stage=False)
    sim.init_equilibrium(*[torch.from_numpy(t).cuda() for t in inputs.smooth_fields(nx, ny, nz, dims=3, seed=1)])
    sim.step(1)
    a = torch.empty(sim.sizes[lbm.BUF_POP_A], dtype=torch.uint8, device="cuda")
    lbm.lbm_save_state(sim.ctx, a, sim.stream)
    b = torch.full_like(a, 0x3C)
    lbm.lbm_step_from(sim.ctx, a, b, 1, sim.stream)
    sim.step(1)
    assert torch.equal(raw(sim, b), raw(sim))
    sim.close()


# with device output the register step runs beside the link sum: the values of
# the two calls in sequence, step after step
@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("box", [(64, 33, 1), (40, 24, 20)])
def test_step_force_beside_the_step(box, storage):
    nx, ny, nz = box
    mask = (inputs.cylinder_mask(nx, ny, (20.2, 16.1), 5.3) if nz == 1 else
            inputs.sphere_mask(nx, ny, nz, (12.2, 11.6, 9.8), 4.4))
    cfg = dict(lattice=9 if nz == 1 else 19, nx=nx, ny=ny, nz=nz, tau=0.7, force_model="e", g=(1e-5, 0, 0),
               storage=storage, wall_u=((0.01, 0, 0),), step_kernel="register")
    a, b = lbm.Sim(cfg, mask), lbm.Sim(cfg, mask)
    n = 200
    ref, got = (torch.zeros((n, 3), dtype=torch.float64, device="cuda") for _ in range(2))
    for s in (a, b):
        s.rest()
        s.step(1)
    for i in range(n):
        lbm.lbm_wall_force(a.ctx, 1, 0, 1.0, ref[i], lbm.OUT_DEVICE, a.stream)
        torch.cuda.synchronize()
        a.step(1)
        torch.cuda.synchronize()
    for i in range(n):
        lbm.lbm_step_force(b.ctx, 1, 0, 1.0, got[i], lbm.OUT_DEVICE, b.stream)
    assert torch.equal(ref, got) and torch.equal(raw(a), raw(b))
    a.close()
    b.close()


# insulating walls on the staged kernel (the automatic choice in FP32): the
# field's mean velocity is summed in another order, so the populations agree to
# a few roundings of FP32 deviations (8 steps of 2^-24 of values below 0.1)
@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("box", [(96, 128, 80), (130, 96, 96)])
def test_insulating_walls_on_the_staged_kernel(box, periodic):
    nx, ny, nz = box
    mask = inputs.sphere_mask(nx, ny, nz, (30.4, 30.2, 24.7), 6.3)
    rho, u = inputs.smooth_fields(nx, ny, nz, dims=3, u_amplitude=0.04, seed=4)
    out = []
    for kernel in ("register", "auto"):
        sim = lbm.Sim(dict(lattice=19, nx=nx, ny=ny, nz=nz, periodic=periodic, tau=0.7, force_model="e",
                           g=(1e-5, 0, 0), lorentz=1, B=(0.0, 0.05, 0.02), sigma_e=1.0, insulating=1, storage="f32",
                           wall_u=((0, 0, 0),), step_kernel=kernel), mask, stage=False)
        assert sim.step_kernel == {"register": "register", "auto": "staged"}[kernel]
        sim.init_equilibrium(torch.from_numpy(rho).cuda(), torch.from_numpy(u).cuda())
        sim.step(8)
        assert sim.device_status() == 0
        out.append((sim.export_f(), sim.electric_field()))
        sim.close()
    assert (out[0][0] - out[1][0]).abs().max() <= 8 * 2.0 ** -24 * 0.1
    assert np.abs(out[0][1] - out[1][1]).max() <= 1e-6 * np.abs(out[0][1]).max()


# the programmatic launches under stream capture: a graph of two steps, the
# second with the force of the first, replayed, against the same calls
@pytest.mark.parametrize("storage,kernel", [("f64", "auto"), ("f32", "register"), ("f16s", "staged")])
def test_steps_in_a_graph(storage, kernel):
    nx, ny, nz = 64, 24, 20
    mask = inputs.sphere_mask(nx, ny, nz, (20.2, 11.6, 9.8), 4.4)
    cfg = dict(lattice=19, nx=nx, ny=ny, nz=nz, tau=0.7, force_model="e", g=(1e-5, 0, 0), storage=storage,
               wall_u=((0.01, 0, 0),), step_kernel=kernel)
    a, b = lbm.Sim(cfg, mask), lbm.Sim(cfg, mask)
    fa, fb = (torch.zeros(3, dtype=torch.float64, device="cuda") for _ in range(2))
    for s in (a, b):
        s.rest()
        s.step(2)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.step(1)
        lbm.lbm_step_force(a.ctx, 1, 0, 1.0, fa, lbm.OUT_DEVICE, a.stream)
    for _ in range(7):
        graph.replay()
        b.step(1)
        lbm.lbm_step_force(b.ctx, 1, 0, 1.0, fb, lbm.OUT_DEVICE, b.stream)
    torch.cuda.synchronize()
    assert torch.equal(fa, fb) and torch.equal(raw(a), raw(b))
    a.close()
    b.close()


def _force_box(name):
    """(configuration, mask, wall distance or None, wall whose force is asked for)"""
    if name == "cavity":           # every face closed, lid moving, Smagorinsky LES
        n = 40
        return dict(nx=n, ny=n, nz=n, periodic=(0, 0, 0), tau=0.55, les=1, cs=0.1, wall_u=((0, 0, 0), (0.1, 0, 0)),
                    face_wall=(1, 1, 1, 1, 1, 2)), inputs.empty_mask(n, n, n), None, 2
    if name == "no_links":         # a wall that no node belongs to
        cfg, mask, _, _ = _force_box("sphere")
        return dict(cfg, wall_u=((0.01, 0, 0), (0, 0, 0))), mask, None, 2
    nx, ny, nz = {"insulating_large": (130, 96, 96)}.get(name, (66, 33, 20))
    centre, r = (20.2, 14.6, 9.8), 4.4
    mask = inputs.sphere_mask(nx, ny, nz, centre, r)
    cfg = dict(nx=nx, ny=ny, nz=nz, tau=0.7, g=(1e-5, 0, 0), wall_u=((0.01, 0, 0),))
    phi = None
    if name == "closed":           # closed in x and z, body force, no EXT terms
        cfg.update(periodic=(0, 1, 0))
    elif name == "les":
        cfg.update(les=1, cs=0.1, tau=0.56)
    elif name == "brinkman":
        cfg.update(stokes=1, darcy=1e-3)
    elif name.startswith("insulating"):
        cfg.update(lorentz=1, B=(0.0, 0.05, 0.02), sigma_e=1.0, insulating=1)
    elif name == "curved":
        z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(float)
        phi = (np.sqrt((x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2) - r).astype(np.float32)
        mask = (phi < 0).astype(np.uint8)
        cfg.update(curved=1)
    return cfg, mask, phi, 1


# lbm_step_force with device output is the wall force and then the step, in
# every box whose force is not summed inside the step kernel: the values of the
# two calls with the device idle in between, step after step
@pytest.mark.parametrize("name,storage,kernel", [
    ("cavity", "f16s", "staged"), ("cavity", "f32", "staged"), ("cavity", "bf16s", "register"), ("cavity", "f64", "auto"),
    ("closed", "f16s", "staged"), ("closed", "f32", "staged"), ("closed", "f64", "auto"),
    ("les", "f16s", "staged"), ("les", "f32", "staged"), ("les", "f16s", "register"),
    ("brinkman", "bf16s", "staged"), ("brinkman", "f32", "staged"), ("brinkman", "f64", "auto"),
    ("insulating", "f32", "register"), ("insulating", "f16s", "auto"), ("insulating", "f64", "auto"),
    ("insulating_large", "f32", "auto"), ("curved", "f32", "auto"), ("curved", "f16s", "auto"), ("curved", "f64", "auto"),
    ("sphere", "f16s", "register"), ("sphere", "bf16s", "register"), ("no_links", "f32", "register"),
    ("no_links", "f16s", "register"), ("no_links", "f64", "auto")])
def test_step_force_with_device_output(name, storage, kernel):
    cfg, mask, phi, wall = _force_box(name)
    cfg = dict(cfg, lattice=19, force_model="e", storage=storage, step_kernel=kernel, seed=3,
               rounding="stochastic" if storage == "f16s" else "nearest")
    a, b = lbm.Sim(cfg, mask), lbm.Sim(cfg, mask)
    if kernel != "auto" or name == "insulating_large":
        assert a.step_kernel == ("staged" if kernel == "auto" else kernel)
    nz, ny, nx = mask.shape
    rho, u = inputs.smooth_fields(nx, ny, nz, dims=3, u_amplitude=0.03, seed=3)
    n = 60
    ref, got = (torch.zeros((n, 3), dtype=torch.float64, device="cuda") for _ in range(2))
    for s in (a, b):
        if phi is not None:
            s.set_wall_distance(phi)
        s.init_equilibrium(rho, u)
        s.step(1)
    torch.cuda.synchronize()
    for i in range(n):
        lbm.lbm_wall_force(a.ctx, wall, 0, 1.0, ref[i], lbm.OUT_DEVICE, a.stream)
        torch.cuda.synchronize()
        a.step(1)
        torch.cuda.synchronize()
    for i in range(n):
        lbm.lbm_step_force(b.ctx, wall, 0, 1.0, got[i], lbm.OUT_DEVICE, b.stream)
    assert torch.equal(ref, got) and torch.equal(raw(a), raw(b))
    assert a.device_status() == 0 and b.device_status() == 0
    assert (name == "no_links") == (not ref.any())
    if name.startswith("insulating"):
        assert np.array_equal(a.electric_field(), b.electric_field())
    a.close()
    b.close()


def load(sim, P, t=0):
    """Make the FP32 array P (Q, nz, ny, nx) the stored post-collision populations."""
    buf = torch.zeros(sim.sizes[lbm.BUF_POP_A], dtype=torch.uint8, device="cuda")
    raw(sim, buf)[..., :sim.shape[2]] = torch.from_numpy(P).cuda()
    lbm.lbm_load_state(sim.ctx, buf, t, sim.stream)
    torch.cuda.synchronize()


# import and export of FP32 populations within a few FP32 steps of the rest
# value w rho0 (a deviation of a few units in the last place of f) and of zero:
# one rounding of the FP64 difference or sum
@pytest.mark.parametrize("rho0", [1.0, 0.7, 3.1, 1.0 / 3.0])
@pytest.mark.parametrize("box", [(64, 7, 1), (64, 3, 5)])
def test_populations_near_rest_are_rounded_once(box, rho0):
    nx, ny, nz = box
    Q = 9 if nz == 1 else 19
    c = W[Q][:, None, None, None] * float(np.float32(rho0))
    sim = lbm.Sim(dict(lattice=Q, nx=nx, ny=ny, nz=nz, tau=0.8, rho0=rho0, force_model="e", storage="f32"),
                  inputs.empty_mask(nx, ny, nz), stage=False)
    steps = np.arange(nx * ny * nz).reshape(nz, ny, nx) - nx * ny * nz // 2
    f = c.astype(np.float32) + steps * np.spacing(c.astype(np.float32))
    sim.import_f(torch.from_numpy(f.astype(np.float32)).cuda())
    P = raw(sim)[..., :nx].cpu().numpy()
    for a in range(Q):                                       # P_a(x) = f_a(x + E_a) - w_a rho0
        d = np.roll(f.astype(np.float32).astype(np.float64) - c, tuple(-E[Q][a][::-1]), axis=(1, 2, 3))[a]
        err = np.abs(P[a].astype(np.float64) - d)
        assert np.all(err <= 0.5 * np.spacing(np.abs(d).astype(np.float32)) * (1 + 2.0 ** -16)), a
    # export: a population near zero, f = d + w rho0 with d near -w rho0
    P = (-c.astype(np.float32) + steps * np.spacing(c.astype(np.float32))).astype(np.float32)
    load(sim, P)
    got = sim.export_f(torch.float32).cpu().numpy()
    for a in range(Q):                                       # f_a(x) = P_a(x - E_a) + w_a rho0
        want = np.roll(P.astype(np.float64) + c, tuple(E[Q][a][::-1]), axis=(1, 2, 3))[a]
        err = np.abs(got[a].astype(np.float64) - want)
        assert np.all(err <= 0.5 * np.spacing(np.abs(want).astype(np.float32)) * (1 + 2.0 ** -16)), a
    sim.close()


# reductions in flight on several streams, which the header forbids, spoil the
# values of those calls alone: the ones after them are right, on every stream,
# also where more streams have been used than have a counter of their own
def test_reductions_after_overlapping_ones():
    nx, ny, nz = 64, 24, 20
    mask = inputs.sphere_mask(nx, ny, nz, (20.2, 11.6, 9.8), 4.4)
    sim = lbm.Sim(dict(lattice=19, nx=nx, ny=ny, nz=nz, tau=0.7, force_model="e", g=(1e-5, 0, 0), storage="f16s",
                       wall_u=((0, 0, 0),), step_kernel="staged"), mask)
    sim.rest()
    sim.step(20)
    v_ref = sim.velocity_buffer()
    scrap = torch.zeros((3, 8), dtype=torch.float64, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(40)]

    def results(stream):
        with torch.cuda.stream(stream):
            force, balance = sim.wall_force(1), sim.balance()
            return np.hstack([force, *balance, sim.residual(v_ref, update=False)])
    torch.cuda.synchronize()
    want = results(streams[0])
    for k in range(0, 36, 3):
        for _ in range(20):
            lbm.lbm_wall_force(sim.ctx, 1, 0, 1.0, scrap[0], lbm.OUT_DEVICE, streams[k].cuda_stream)
            lbm.lbm_balance(sim.ctx, scrap[1], lbm.OUT_DEVICE, streams[k + 1].cuda_stream)
            lbm.lbm_residual(sim.ctx, v_ref, False, scrap[2], lbm.OUT_DEVICE, streams[k + 2].cuda_stream)
        torch.cuda.synchronize()
        for stream in (streams[k], streams[k + 1], streams[k + 2], streams[39]):
            assert np.array_equal(results(stream), want)
    got = np.zeros(3)
    lbm.lbm_step_force(sim.ctx, 1, 0, 1.0, got, lbm.OUT_HOST, sim.stream)
    assert np.abs(got - want[:3]).max() <= 1e-12 * np.abs(want[:3]).max()
    sim.close()


# ... with rows that end one node into a pitch, in its last chunk, and of one node
@pytest.mark.parametrize("storage", ["f32", "f16s"])
@pytest.mark.parametrize("nx", [1, 61, 63, 65, 124])
def test_step_from_leaves_no_padding_at_row_ends(nx, storage):
    test_step_from_leaves_no_padding(nx, storage, "staged")
