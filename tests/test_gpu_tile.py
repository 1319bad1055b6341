"""The tile schedules (one launch per timestep on lattices too small for the march), which AUTO
picks by size: against the FP64 oracle at the edges of their tiles -- lattices smaller than a
tile, exact multiples, remainders of one -- with every term on, between walls and under the
Gibbs-Duhem form, and against the other schedules' ghost columns by bands."""
import numpy as np
import pytest

import paper_0704_3444_gb300 as mclb
from oracle import Oracle
from paper_0704_3444_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    mclb.build()
    mclb.load()


def _pair(shape, precision, fv=0, walls=0, gd=0, amp=0.3, seed=70):
    nx, ny, n = shape
    rho, u = inputs.random_state(n, nx, ny, seed=seed + nx + n, amp=amp, umax=0.03)
    chi = inputs.uniform_chi(n, 1.6)
    kw = dict(m=[1.0 + (k % 3) for k in range(n)], theta=0.4, kappa=0.0 if gd else 0.02,
              force=(1e-5, -2e-5), forcing_velocity=fv, walls=walls, force_form=gd)
    sim = mclb.Simulation(n, nx, ny, 0.9, chi, precision=precision, **kw)
    orc = Oracle(n, nx, ny, 0.9, chi, **kw)
    sim.init_fields(rho, u)
    orc.init(rho, u)
    return sim, orc


def _rel(a, b):
    return np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300)


SHAPES = [(1, 1, 2), (4, 4, 2), (1, 9, 3), (9, 1, 1), (5, 3, 3), (8, 4, 5), (9, 5, 6), (33, 13, 8),
          (130, 100, 4), (161, 97, 2)]


@pytest.mark.parametrize("mode", ["periodic", "barycentric", "walls", "gibbs_duhem"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[0]}x{s[1]}N{s[2]}")
def test_fp64_parity(shape, mode):
    """40 FP64 steps (one graph of 32 and 8 more) to the oracle parity of the other
    schedules (1e-12 of the field's max-norm)."""
    gd = mode == "gibbs_duhem"
    if gd and shape[2] > 3:
        pytest.skip("the form runs staged there")
    sim, orc = _pair(shape, "fp64", fv=int(mode != "periodic"), walls=int(mode == "walls"), gd=int(gd))
    assert sim.launches_per_step == (2 if gd else 1)
    sim.step(40)
    assert orc.run(40) == 0
    assert sim.status() == 0
    assert _rel(sim.get_state(), orc.f) < 1e-12
    # the ghost columns are the columns they repeat: a schedule that reads them goes on from
    # the same stored rows
    nx, ny, n = shape
    if mode != "walls":
        import torch
        band = torch.empty(sim.rows_bytes(ny) // 8, dtype=torch.float64, device="cuda")
        sim.pack_rows(0, ny, band)
        fused = mclb.Simulation(n, nx, ny, 0.9, inputs.uniform_chi(n, 1.6), precision="fp64",
                                kernel=mclb.KERNEL_FUSED, m=[1.0 + (k % 3) for k in range(n)], theta=0.4,
                                kappa=0.0 if gd else 0.02, force=(1e-5, -2e-5),
                                forcing_velocity=int(mode != "periodic"), force_form=int(gd))
        torch.cuda.synchronize()
        fused.unpack_rows(0, ny, band)
        fused.step(3)
        orc.run(3)
        assert _rel(fused.get_state(), orc.f) < 1e-12
        fused.close()
    sim.close()


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("shape", [(37, 21, 3), (16, 8, 1), (400, 190, 2), (279, 181, 3), (29, 5600, 1), (420, 160, 4),
                                   (225, 200, 5), (90, 70, 8)],
                         ids=lambda s: f"{s[0]}x{s[1]}N{s[2]}")
def test_fp32_parity(shape, walls):
    """100 FP32 steps: rho, U and mu within the FP32 tolerance of the fields (1e-5)."""
    sim, orc = _pair(shape, "fp32", walls=walls, amp=0.1)
    assert sim.launches_per_step == 1
    sim.step(100)
    assert orc.run(100) == 0
    assert sim.status() == 0
    gm, om = sim.moments(), orc.moments()
    for k in ("rho", "U", "mu"):
        assert np.max(np.abs(gm[k] - om[k])) < 1e-5, k
    sim.close()


@pytest.mark.parametrize("precision", ["bf16", "fp16"])
@pytest.mark.parametrize("shape,walls", [((37, 21, 3), 0), ((150, 61, 4), 1), ((16, 8, 6), 0)],
                         ids=["37x21N3", "150x61N4walls", "16x8N6"])
def test_16_bit_parity(shape, walls, precision):
    """The 16-bit formats: densities within 2e-3 and every component's mass to 1e-6, as the
    other schedules keep them."""
    sim, orc = _pair(shape, precision, walls=walls, amp=0.1)
    assert sim.launches_per_step == 1
    m0 = sim.conservation()["mass"]
    sim.step(50)
    assert orc.run(50) == 0
    assert sim.status() == 0
    assert np.max(np.abs(sim.moments()["rho"] - orc.moments()["rho"])) < 2e-3
    assert np.max(np.abs(sim.conservation()["mass"] / m0 - 1.0)) < 1e-6
    sim.close()


@pytest.mark.parametrize("precision,shape", [("fp64", (50, 40, 2)), ("fp32", (50, 40, 2)), ("fp32", (300, 190, 3))])
def test_resume_and_non_finite(precision, shape):
    """A state read back and set again goes on bitwise; a density that turns non-finite is
    reported."""
    sim, _ = _pair(shape, precision)
    sim.step(35)
    mid = sim.get_state()
    sim.step(33)
    end = sim.get_state()
    sim.set_state(mid)
    sim.step(33)
    assert np.array_equal(sim.get_state(), end)
    assert sim.status() == 0
    mid[:] = -mid
    sim.set_state(mid)
    sim.step_nocheck(1)
    assert sim.status() == -4
    sim.close()


def test_fp32_batch_by_row_tiles():
    """FP32 batches large enough for the row tiles: instances narrower than a tile, at exact
    multiples and with remainders, two groups side by side, an odd and an even number of
    steps; densities and U within the FP32 tolerance of the oracle (1e-5) after 41 steps,
    and the march takes over the same state from the tiles' ghost columns."""
    probs = []
    for k, (nx, ny, n) in enumerate([(700, 500, 2), (28, 12, 2), (421, 403, 2), (650, 433, 3), (57, 16, 3), (280, 240, 3)]):
        rho, u = inputs.random_state(n, nx, ny, seed=640 + k, amp=0.1, umax=0.03)
        p = inputs.Problem(name=f"r{k}", ncomp=n, nx=nx, ny=ny, tau=0.7 + 0.1 * k, chi=inputs.uniform_chi(n, 1.7),
                           m=np.ones(n), theta=1 / 3, kappa=0.01, force=(1e-5, 0.0), rho=rho, u=u)
        p.forcing_velocity = k % 2
        probs.append(p)
    b = mclb.Batch(probs, precision="fp32")
    b.init_all()
    b.step(1)
    assert [w for _, w in b.tuning()] == [1, 1] and b.launches_per_step == 2
    b.step(40)
    assert b.status()[0] == 0
    oracles = []
    for k, p in enumerate(probs):
        orc = Oracle.from_problem(p)
        orc.run(41)
        oracles.append(orc)
        got, want = b.moments(k), orc.moments()
        for f in ("rho", "U"):
            assert np.max(np.abs(got[f] - want[f])) < 1e-5, (k, f)
    assert b.test_force_partition(False, 4) == 2
    b.step(3)
    for k in (1, 4, 5):
        oracles[k].run(3)
        assert np.max(np.abs(b.moments(k)["rho"] - oracles[k].moments()["rho"])) < 1e-5, k
    b.close()


@pytest.mark.parametrize("precision,shape,steps", [("fp32", (1500, 601, 3), 10), ("bf16", (701, 420, 3), 10),
                                                   ("fp64", (1003, 760, 4), 5), ("fp32", (420000, 6, 1), 6)],
                         ids=lambda v: str(v))
def test_march_between_walls_with_wall_tiles(precision, shape, steps):
    """Lattices between walls that the march steps under AUTO: the rows next to the walls by one
    tile launch; densities, U (and the FP64 state) to the formats' parity with the oracle."""
    sim, orc = _pair(shape, precision, fv=1, walls=1, amp=0.1)
    assert sim.launches_per_step == 3
    sim.step(steps)
    assert orc.run(steps) == 0
    assert sim.status() == 0
    got, want = sim.moments(mu=False, P=False), orc.moments()
    tol = {"fp64": 1e-12, "fp32": 1e-5, "bf16": 2e-3}[precision]
    assert np.max(np.abs(got["rho"] - want["rho"])) < tol and np.max(np.abs(got["U"] - want["U"])) < tol
    if precision == "fp64":
        assert _rel(sim.get_state(), orc.f) < 1e-12
    sim.close()


def test_fp32_batch_of_tiles_and_march():
    """One group by row tiles and one, of few large instances, by the march: one after the other on
    one stream, densities and U within the FP32 tolerance of the oracle (1e-5) after 35 steps (a
    replayed graph and single steps)."""
    probs = []
    for k, (nx, ny, n) in enumerate([(700, 720, 2), (400, 423, 3), (409, 420, 3)]):
        rho, u = inputs.random_state(n, nx, ny, seed=660 + k, amp=0.1, umax=0.03)
        probs.append(inputs.Problem(name=f"m{k}", ncomp=n, nx=nx, ny=ny, tau=0.8 + 0.1 * k, chi=inputs.uniform_chi(n, 1.7),
                                    m=np.ones(n), theta=1 / 3, kappa=0.01, force=(1e-5, 0.0), rho=rho, u=u))
    b = mclb.Batch(probs, precision="fp32")
    b.init_all()
    b.step(35)
    waves = [w for _, w in b.tuning()]
    assert waves[0] == 1 and waves[1] in (2, 4, 8, 16) and b.launches_per_step == 3
    assert b.status()[0] == 0
    for k, p in enumerate(probs):
        orc = Oracle.from_problem(p)
        orc.run(35)
        got, want = b.moments(k), orc.moments()
        for f in ("rho", "U"):
            assert np.max(np.abs(got[f] - want[f])) < 1e-5, (k, f)
    b.close()


SHAPES_16 = [(1, 1, 1, 0), (5, 9, 2, 0), (37, 21, 3, 0), (64, 64, 4, 0), (300, 170, 4, 0), (61, 47, 5, 0), (90, 33, 6, 0),
             (41, 30, 7, 0), (16, 8, 8, 0), (130, 1, 2, 1), (17, 3, 1, 1), (33, 4, 3, 1), (20, 6, 2, 1), (50, 7, 4, 1),
             (150, 61, 4, 1), (29, 14, 5, 1), (45, 23, 6, 1), (18, 15, 7, 1), (9, 40, 8, 1), (701, 420, 3, 1),
             (1003, 310, 5, 1)]


@pytest.mark.parametrize("precision", ["bf16", "fp16"])
@pytest.mark.parametrize("shape", SHAPES_16, ids=lambda s: f"{s[0]}x{s[1]}N{s[2]}" + ("walls" if s[3] else ""))
def test_16_bit_schedules_agree(shape, precision):
    """Which schedule steps a 16-bit lattice does not show: after 50 steps the state of AUTO (tiles, or
    the march with the rows next to walls by tiles) is that of FUSED bit for bit, ghost columns included."""
    import torch
    nx, ny, n, walls = shape
    rho, u = inputs.random_state(n, nx, ny, seed=90 + nx + n, amp=0.3, umax=0.05)
    x = np.random.default_rng(n).uniform(0.5, 2.0, (n, n))
    kw = dict(m=[1.0 + (k % 3) * (nx % 2) for k in range(n)], theta=0.4 if ny % 2 else 1 / 3, kappa=0.02,
              force=(1e-5, -2e-5), forcing_velocity=n // 2 % 2)
    chi = np.triu(x, 1) + np.triu(x, 1).T
    got = {}
    for kernel in (mclb.KERNEL_AUTO, mclb.KERNEL_FUSED):
        sim = mclb.Simulation(n, nx, ny, 0.9, chi, precision=precision, kernel=kernel, walls=walls, **kw)
        sim.init_fields(rho, u)
        sim.step(50)
        assert sim.status() == 0
        raw = torch.zeros(sim.rows_bytes(ny), dtype=torch.uint8, device="cuda")
        sim.pack_rows(0, ny, raw)
        got[kernel] = (sim.get_state(), sim.moments(mu=False, P=False)["U"], raw.cpu().numpy(), sim.launches_per_step)
        sim.close()
    auto, fused = got[mclb.KERNEL_AUTO], got[mclb.KERNEL_FUSED]
    assert auto[3] < fused[3]
    for a, b in zip(auto[:3], fused[:3]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("precision,shape,walls,launches", [
    ("fp64", (690, 700, 4), 0, 1), ("fp64", (800, 800, 4), 0, 2), ("fp64", (560, 560, 5), 0, 1),
    ("fp64", (770, 770, 5), 0, 2), ("fp64", (700, 690, 5), 1, 1), ("fp64", (760, 760, 5), 1, 3),
    ("fp64", (900, 900, 6), 0, 1), ("fp32", (1500, 1500, 1), 1, 1), ("fp32", (1050, 1050, 2), 1, 3),
    ("fp32", (800, 800, 3), 1, 1), ("fp32", (785, 785, 4), 1, 3), ("fp32", (700, 700, 5), 1, 3),
    ("fp32", (300, 350, 6), 1, 1), ("fp32", (500, 500, 6), 1, 3), ("fp32", (400, 400, 7), 1, 3),
    ("fp32", (300, 300, 8), 1, 1), ("fp32", (400, 400, 8), 1, 3)], ids=str)
def test_auto_takes_the_faster_schedule(precision, shape, walls, launches):
    """On both sides of the lines where tiles and march measured equal: one launch a step is the
    tiles, two (three between walls) the march."""
    nx, ny, n = shape
    sim = mclb.Simulation(n, nx, ny, 0.9, inputs.uniform_chi(n, 1.6), precision=precision, walls=walls)
    assert sim.launches_per_step == launches
    sim.close()


@pytest.mark.parametrize("n,edge,launches", [(1, 128, 3), (1, 224, 2), (2, 96, 2), (4, 96, 3), (4, 128, 2)])
def test_auto_takes_the_faster_d3q19_schedule(n, edge, launches):
    """As above: three launches a step are the staged step, two the march; the fields are those of
    the other schedule bit for bit."""
    import torch
    rho = 1.0 / n + 0.02 * torch.rand(n, edge, edge, edge, generator=torch.Generator("cuda").manual_seed(n),
                                      dtype=torch.float64, device="cuda")
    u = torch.zeros(3, edge, edge, edge, dtype=torch.float64, device="cuda")
    got = []
    for kernel in (mclb.KERNEL_AUTO, mclb.KERNEL_STAGED if launches == 2 else mclb.KERNEL_FUSED):
        sim = mclb.Simulation(n, edge, edge, 0.9, inputs.uniform_chi(n, 1.6), precision="fp32", lattice="d3q19",
                              nz=edge, kappa=0.02, kernel=kernel)
        assert sim.launches_per_step == (launches if kernel == mclb.KERNEL_AUTO else 5 - launches)
        r, v = rho.clone(), u.clone()
        sim.init_fields_device(r, v)
        torch.cuda.synchronize()
        sim.step(3)
        sim.moments_device(rho=r, U=v)
        assert sim.status() == 0
        got.append((r.cpu(), v.cpu()))
        sim.close()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("n,sizes", [
    (1, [(160, 97), (1, 1), (33, 40)]), (2, [(128, 104), (130, 61), (17, 9)]), (3, [(16, 8), (121, 113), (5, 3)]),
    (6, [(64, 48), (67, 35), (4, 9)]), (8, [(24, 12), (41, 30)])], ids=lambda v: str(v) if isinstance(v, int) else "")
def test_fp64_batch_by_tiles(n, sizes):
    """FP64 batches by tiles of 16 x 8 (more than 12800 sites in all) and of 8 x 4 sites (five and more
    components), exact multiples and remainders: every state within 1e-12 of the oracle after a
    replayed graph of 32 steps and nine more."""
    probs = []
    for k, (nx, ny) in enumerate(sizes):
        rho, u = inputs.random_state(n, nx, ny, seed=680 + k, amp=0.3, umax=0.02)
        p = inputs.Problem(name=f"f{k}", ncomp=n, nx=nx, ny=ny, tau=0.8 + 0.1 * k, chi=inputs.uniform_chi(n, 1.6),
                           m=np.array([1.0 + (s % 3) for s in range(n)]), theta=0.4, kappa=0.02, force=(1e-5, -2e-5),
                           rho=rho, u=u)
        p.forcing_velocity = k % 2
        probs.append(p)
    b = mclb.Batch(probs, precision="fp64")
    b.init_all()
    b.step(41)
    assert [w for _, w in b.tuning()] == [1] and b.launches_per_step == 2
    assert b.status()[0] == 0
    for k, p in enumerate(probs):
        orc = Oracle.from_problem(p)
        assert orc.run(41) == 0
        assert _rel(b.get_state(k), orc.f) < 1e-12, k
    b.close()
