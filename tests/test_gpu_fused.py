"""The kernels that take several D2Q9 steps per launch (launch vec 10, 11, 12 and
the default) against the one-step kernel, bit for bit: they run the same
operations in the same order, so the whole state has to be equal, at the edges
of their strips, tiles and row ranges, for every wall kind, velocity kind,
storage form and alignment."""
import numpy as np
import pytest
import torch

from _common import Case, assert_parity, run_oracle
from paper_1404_2363_gb300.solver import Solver

pytestmark = pytest.mark.gpu

# nx: below, at and past the 56 columns of a strip and the 48 .. 60 of a tile; multiples of 8, 4 and 2, and odd
# (16-byte copies, paired stores, neither). ny: fewer rows than the halo of eight, tile remainders, several ranges
SIZES = [(5, 3), (8, 9), (56, 129), (57, 21), (64, 40), (127, 18), (300, 37), (114, 70)]
Y = [("periodic", "periodic"), ("noflux", "bounceback"), ("bounceback", "noflux"), ("dirichlet", "bounceback"),
     ("noflux", "dirichlet")]
X = [("periodic", "periodic"), ("noflux", "bounceback"), ("bounceback", "noflux")]


def state(case, shape, steps):
    s = Solver(nx=case.nx, ny=case.ny, storage=case.storage, bc=case.bc, bc_x=case.bc_x, phi_w=case.phi_w,
               model=case.model)
    if shape is not None:
        s.set_launch(*shape)
    s.set_D(case.D)
    phi0, a, sched = case.inputs()
    if a is not None:
        s.set_velocity(torch.from_numpy(a).cuda(), None if sched is None else torch.from_numpy(sched).cuda(),
                       kind="row" if case.ukind == "row" else "field")
    s.set_phi(torch.from_numpy(phi0).cuda())
    for n in steps:
        s.step(n)
    g, t = s.get_state()
    g = g.cpu().numpy()
    s.close()
    assert t == sum(steps)
    return g


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_fused_steps_equal_single_steps(storage, nx, ny):
    for j, (bc, bx) in enumerate((bc, bx) for bc in Y for bx in X):
        uk = ("field", "row", "none")[j % 3] if bx[0] == "periodic" else "field"
        model = ("A", "B1", "B3")[j % 3] if storage == "f32" and "dirichlet" not in bc else "A"
        case = Case(nx=nx, ny=ny, storage=storage, bc=bc, bc_x=bx, ukind=uk, phi_w=(0.7, 0.3), model=model, umax=0.02)
        ref = state(case, (128, 1), [15])      # 8 + 7, 4 x 3 + 2 + 1
        for shape in ((128, 11), (128, 12), None):
            got = state(case, shape, [15])
            assert np.array_equal(got, ref), (shape, bc, bx, uk, model)


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_fused_steps_do_not_depend_on_their_grouping(storage):
    case = Case(nx=200, ny=61, storage=storage)
    ref = state(case, (128, 1), [41])
    for shape in ((128, 11), (128, 12), (128, 10), None):
        for steps in ([41], [1] * 5 + [2, 3, 4, 5, 6, 7, 9], [40, 1], [8, 33]):
            assert np.array_equal(state(case, shape, steps), ref), (shape, steps)


@pytest.mark.parametrize("shape", [(128, 11), (128, 12)])
def test_fused_steps_match_oracle(O, shape):
    case = Case(nx=181, ny=53, steps=120, bc=("noflux", "bounceback"), bc_x=("bounceback", "noflux"))
    phi0, a, sched = case.inputs()
    g = state(case, shape, [case.steps]).view(np.float32).reshape(9, case.ny, case.nx)
    assert_parity(g.astype(np.float64).sum(0), run_oracle(O, case, phi0, a, sched), 1e-5)


def test_fused_steps_on_an_unaligned_velocity_field():
    """A velocity field that starts 4 bytes past a 16-byte boundary: no 16-byte copies, the same state."""
    nx, ny = 112, 40
    case = Case(nx=nx, ny=ny, sched=False)
    phi0, a, _ = case.inputs()
    buf = torch.zeros(2 * nx * ny + 1, device="cuda")
    buf[1:] = torch.from_numpy(a).cuda().reshape(-1)
    out = []
    for shape in ((128, 1), (128, 11), (128, 12)):
        s = Solver(nx=nx, ny=ny)
        s.set_launch(*shape)
        s.set_D(case.D)
        s.set_velocity(buf[1:].reshape(2, ny, nx))
        s.set_phi(torch.from_numpy(phi0).cuda())
        s.step(14)
        out.append(s.get_state()[0].cpu().numpy())
        s.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


def test_fused_launch_shapes_are_checked():
    from paper_1404_2363_gb300 import _native as N

    s = Solver(lattice=15, nx=16, ny=16, nz=4)
    for vec in (10, 11, 12):
        with pytest.raises(N.LbmError):
            s.set_launch(128, vec)
    s.close()
    s = Solver(nx=16, ny=16)
    for block, vec in ((256, 10), (128, 0), (128, 13)):
        with pytest.raises(N.LbmError):
            s.set_launch(block, vec)
    s.close()


def test_batch_walk_equals_one_step_launches():
    """Several batch steps per launch (PER_STEP mode on batches large enough for it) against the persistent
    cell tiles, which take one step at a time: fields and moments bit for bit, over odd and even row lengths,
    heights off the 16-row tiles, every wall pair and model, with and without a velocity; 21 steps are two
    groups of eight and five single ones, in chunks of 16."""
    from paper_1404_2363_gb300.batch import Batch, poiseuille_row

    g = np.random.default_rng(5)
    walls = [("noflux", "noflux"), ("bounceback", "bounceback"), ("periodic", "periodic"), ("noflux", "bounceback"),
             ("bounceback", "noflux")]
    chs, phis = [], []
    for i in range(48):
        nx, ny = int(g.integers(1500, 2600)), int(g.integers(30, 90))
        chs.append({"nx": nx, "ny": ny, "bc": walls[i % 5], "D": [[0.03, 0.004], [0.004, 0.05]],
                    "u_row": poiseuille_row(ny, 0.08) if i % 7 else None, "x_ref0": float(round(0.2 * nx)),
                    "x_ref_velocity": 0.05, "model": ("A", "B1", "B2", "B3")[i % 4]})
        phis.append((0.05 + g.random((ny, nx))).astype(np.float32))
    out = []
    for mode in ("persistent", "per_step"):
        b = Batch(chs, mode=mode, tile_rows=0, graph_steps=16)
        b.set_phi(phis)
        m = b.run(21)
        out.append((m, torch.cat([p.reshape(-1) for p in b.get_phi()])))
        b.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("lattice,storage,launch", [
    (15, "f32", (64, 1)), (15, "f16", (64, 1)), (15, "bf16", (64, 1)), (15, "bf16", (64, 5)), (15, "f16", (128, 9)),
    (9, "f32", (64, 1)), (9, "bf16", (64, 1)), (9, "f32", (128, 11)), (9, "f16", (128, 12)), (9, "f32", None)])
def test_overlapping_launches_equal_separate_ones(lattice, storage, launch):
    """Each launch may start while the one before it drains: many launches in a row on a grid small enough for
    several to be resident at once, against the same launches with the stream drained after each."""
    kw = dict(nx=64, ny=24, nz=20, bc_z=("periodic", "periodic")) if lattice == 15 else dict(nx=192, ny=60)
    D = np.array([[0.03, 0.005, -0.004], [0.005, 0.025, 0.003], [-0.004, 0.003, 0.035]])
    case = Case(lattice=lattice, storage=storage, bc=("noflux", "noflux"), ukind="row", **kw)
    phi0, a, sched = case.inputs()
    chunk = 8 if launch is None or launch[1] > 10 else 1
    out = []
    for wait in (True, False):
        s = Solver(lattice=lattice, nx=case.nx, ny=case.ny, nz=case.nz, storage=storage, bc=case.bc)
        if launch is not None:
            s.set_launch(*launch)
        s.set_D(D if lattice == 15 else case.D)
        s.set_velocity(torch.from_numpy(a).cuda(), torch.from_numpy(sched).cuda(), kind="row")
        s.set_phi(torch.from_numpy(phi0).cuda())
        if wait:
            for _ in range(400 // chunk):
                s.step(chunk)
                torch.cuda.synchronize()
        else:
            s.step(400)
        out.append(s.get_state()[0].cpu().numpy())
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("nx,ny,nz,ukind,shape", [
    (64, 225, 74, "field", (32, 5)), (96, 133, 90, "field", (96, 1)), (200, 101, 53, "field", (128, 5)),
    (200, 101, 53, "none", (224, 1)), (64, 128, 130, "none", (128, 9)), (64, 128, 130, "field", (128, 9))])
def test_default_d3q15_16bit_kernel(nx, ny, nz, ukind, shape):
    """The default of the D3Q15 16-bit forms from 2^20 nodes on: the bits of the kernel that the rule on the row
    length and the velocity names (one node per thread gives its bits with any block)."""
    g = np.random.default_rng(3)
    phi0 = torch.from_numpy((0.5 + 0.1 * g.random((nz, ny, nx))).astype(np.float32)).cuda()
    a = torch.from_numpy((0.05 * g.random((3, nz, ny, nx)) - 0.025).astype(np.float32)).cuda()
    out = []
    for launch in (None, shape):
        s = Solver(lattice=15, nx=nx, ny=ny, nz=nz, storage="bf16")
        if launch is not None:
            s.set_launch(*launch)
        s.set_D([[0.03, 0.005, -0.004], [0.005, 0.025, 0.003], [-0.004, 0.003, 0.035]])
        if ukind == "field":
            s.set_velocity(a)
        s.set_phi(phi0)
        s.step(6)
        out.append(s.get_state()[0].cpu().numpy())
        s.close()
    assert np.array_equal(out[0], out[1])
