"""The walk kernel where its ranges hold several rows (a warp passes from the instance of the wall rows to the plain
one and back, strips with an x wall have ranges of their own), and its instances that store the states between for the
reverse sweep: bit for bit the states and gradients of single steps."""
import numpy as np
import pytest
import torch

from paper_1404_2363_gb300.solver import Solver

pytestmark = pytest.mark.gpu

D = np.array([[0.03, 0.004], [0.004, 0.05]])
Y = [("periodic", "periodic"), ("noflux", "bounceback"), ("bounceback", "noflux"), ("dirichlet", "bounceback"),
     ("noflux", "dirichlet"), ("bounceback", "bounceback")]
X = [("periodic", "periodic"), ("noflux", "bounceback"), ("bounceback", "noflux"), ("noflux", "noflux")]


def make(nx, ny, storage, bc, bc_x, u, seed=29):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = Solver(nx=nx, ny=ny, storage=storage, bc=bc, bc_x=bc_x, phi_w=(0.7, 0.3))
    s.set_D(D)
    a = None
    if u != "none":
        a = 0.04 * torch.rand((2, ny, nx) if u == "field" else (2, ny), device="cuda", generator=g) - 0.02
        s.set_velocity(a, torch.rand((7, 2), device="cuda", generator=g), kind=u)
    return s, 0.1 + torch.rand((ny, nx), device="cuda", generator=g), torch.rand((ny, nx), device="cuda", generator=g)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(704, 900), (702, 650), (701, 830), (60, 20011), (113, 9001)])
def test_ranges_of_several_rows(storage, nx, ny):
    """At 8 warps per SM 13 strips have at most 93 ranges: 7 to 10 rows each; two strips 608, three 405."""
    for j, (bc, bx) in enumerate((bc, bx) for bc in Y for bx in X):
        u = ("field", "row", "none")[j % 3] if bx[0] == "periodic" else ("field", "none")[j % 2]
        state = []
        for launch in ((128, 1), (128, 11)):
            s, phi0, _ = make(nx, ny, storage, bc, bx, u)
            s.set_launch(*launch)
            s.set_phi(phi0)
            s.step(11)                   # 4 + 4 + 2 + 1
            state.append(s.get_state()[0])
            s.close()
        assert torch.equal(*state), (bc, bx, u)


@pytest.mark.parametrize("nx,ny", [(704, 620), (702, 601), (701, 611)])
def test_gradients_do_not_depend_on_the_recompute(nx, ny):
    """Checkpoints every 7 steps of 20 (recompute of 4 + 2 steps), every step and one for all; walls, row lengths
    (16-byte copies, paired stores, neither) and velocities."""
    for j, (bc, bx) in enumerate((bc, bx) for bc in Y[:5] for bx in X[:3]):
        u = ("field", "row", "none")[j % 3] if bx[0] == "periodic" else ("field", "none")[j % 2]
        da = u == "field" and "dirichlet" not in bc
        ref = None
        for launch, every in (((128, 1), 7), ((128, 11), 7), ((128, 12), 7), ((128, 11), 20), ((128, 11), 1), (None, 7)):
            s, phi0, g = make(nx, ny, "f32", bc, bx, u)
            if launch is not None:
                s.set_launch(*launch)
            phi = s.forward_ckpt(phi0, 20, every=every)
            dphi0, dD, ds, du = s.backward(g, want_da=da)
            got = [phi, dphi0, torch.from_numpy(dD.copy()), torch.from_numpy(ds.copy())] + ([du] if da else [])
            s.close()
            if ref is None:
                ref = got
            # sums of slices follow the segments: dD and ds bitwise only with equal checkpoints
            same = range(len(got)) if every == 7 else [0, 1] + ([4] if da else [])
            assert all(torch.equal(got[k], ref[k]) for k in same), (bc, bx, u, launch, every)
