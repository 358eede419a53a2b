"""The passes over a finished state (loss and its seed, macroscopic fields, permeability) and the last launch
of a sweep, at the sizes where their node lists, chunk lengths and grids change: less than a chunk, ragged
ends, every chunk length, more chunks than blocks, no fluid node in a chunk.  The reference is the same sums
over whole arrays in FP64."""
import pytest
import torch

from oracle import oracle as O
from paper_2310_00810_gb300 import lbm

pytestmark = pytest.mark.gpu

SIZES = [(9, 37, 5, 1), (9, 130, 127, 1), (9, 512, 257, 1), (9, 700, 401, 1), (9, 1100, 1021, 1),
         (19, 9, 7, 5), (19, 40, 33, 31), (19, 96, 90, 65)]


def _case(q, nx, ny, nz, precision, **kw):
    g = torch.Generator(device="cuda").manual_seed(nx * 7 + q)
    shape = (ny, nx) if q == 9 else (nz, ny, nx)
    mask = (torch.rand(shape, generator=g, device="cuda") < 0.5).to(torch.uint8)
    mask.view(-1)[: mask.numel() // 3] = 1  # chunks without a fluid node
    mask[..., 0] = 0
    mask[..., -1] = 0
    s = lbm.Solver(q, nx, ny, nz, precision=precision, geometry=mask.cpu(), **kw)
    f = (torch.rand((q, *shape), generator=g, device="cuda", dtype=torch.float64) - 0.4) * 1e-2
    f = (f * (mask == 0)).to(s.plan.dtype)
    ut = (torch.rand((s.plan.d, *shape), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 1e-2
    roi = (torch.rand(shape, generator=g, device="cuda") < 0.7).to(torch.uint8)
    c = torch.as_tensor(O.lattice(q)[0].astype("float64"), device="cuda")[:, : s.plan.d]
    fd = f.double()
    rho = 1.0 + fd.sum(0)
    u = torch.einsum("ka,k...->a...", c, fd) / rho
    return s, mask == 0, f, ut, roi, c, rho, u


def _rel(a, b):
    return ((a - b).norm() / b.norm()).item()


@pytest.mark.parametrize("precision", [4, 8])
@pytest.mark.parametrize("size", SIZES)
def test_macroscopic_and_darcy(size, precision):
    q, nx, ny, nz = size
    s, fl, f, ut, roi, c, rho, u = _case(*size, precision)
    rg, ug = s.macroscopic(f)
    # FP64 throughout: the sum of q terms and one quotient
    assert _rel(rg, rho * fl) < 1e-14 and _rel(ug, u * fl) < 1e-13
    assert not ug[:, ~fl].any() and not rg[~fl].any()
    xs = nx - 1
    rin = torch.tensor([1.01], dtype=torch.float64, device="cuda")
    tau = torch.tensor([0.8], dtype=torch.float64, device="cuda")
    k, flux = s.darcy(f, rin, tau, 1.0, xs)
    J = (u[0] * rho * fl)[..., xs].sum() / (ny * nz)
    dpdx = 0.01 / (3 * nx)
    # terms of both signs: the sum is held to its terms, not to itself
    tol = 1e-13 * (u[0] * rho * fl)[..., xs].abs().sum().item() / (ny * nz)
    assert abs(flux.item() - J.item()) <= tol
    assert abs(k.item() - 0.1 * J.item() / dpdx) <= 0.1 / dpdx * (tol + 1e-12 * abs(J.item()))


@pytest.mark.parametrize("kind", [lbm.LBM_LOSS_VEC, lbm.LBM_LOSS_NORM])
@pytest.mark.parametrize("norm", [lbm.LBM_NORM_SUM, lbm.LBM_NORM_MEAN_FLUID])
@pytest.mark.parametrize("size", SIZES[1:5:3] + SIZES[6:7])
def test_loss_and_seed(size, kind, norm):
    s, fl, f, ut, roi, c, rho, u = _case(*size, 8, loss_kind=kind, loss_norm=norm)
    for r in (None, roi):
        on = fl if r is None else fl & (r != 0)
        lam = torch.full_like(f, float("nan"))
        L, lam = s.loss_grad(f, ut, r, lam=lam)
        w = 1.0 / on.sum().item() if norm == lbm.LBM_NORM_MEAN_FLUID else 1.0
        if kind == lbm.LBM_LOSS_VEC:
            e2, du = ((u - ut) ** 2).sum(0), 2 * w * (u - ut)
        else:
            e = u.norm(dim=0) - ut.norm(dim=0)
            e2, du = e * e, 2 * w * e * u / u.norm(dim=0).clamp_min(1e-300)
        want = torch.einsum("a...,ka->k...", du, c) - (du * u).sum(0)
        want = torch.where(on, want / rho, torch.zeros_like(want))
        # FP64 with sums of a few terms of one size per node; the norm's e cancels a digit or two
        assert abs(L.item() - w * e2[on].sum().item()) <= 1e-11 * L.item()
        assert _rel(lam, want) < 1e-11
        assert not lam[:, ~on].any()


@pytest.mark.parametrize("q,nx,ny,nz", [(9, 33, 9, 1), (19, 31, 6, 5)])
@pytest.mark.parametrize("precision", [4, 8])
@pytest.mark.parametrize("steps", [1, 2, 5])
def test_last_launch_writes_every_entry(q, nx, ny, nz, precision, steps):
    """Whatever the caller's array holds: the fluid-only sweep leaves the dense layout's state, zeros included."""
    g = torch.Generator().manual_seed(3)
    shape = (ny, nx) if q == 9 else (nz, ny, nx)
    mask = (torch.rand(shape, generator=g) < 0.4).to(torch.uint8)
    rin = torch.tensor([1.01], dtype=torch.float64, device="cuda")
    tau = torch.tensor([0.8], dtype=torch.float64, device="cuda")
    out = []
    for layout in ("compact", "dense"):
        s = lbm.Solver(q, nx, ny, nz, precision=precision, n_steps=steps, geometry=mask, layout=layout)
        f = torch.full((q, *shape), float("nan"), device="cuda", dtype=s.plan.dtype)
        out.append(s.forward(rin, tau, 1.0, f=f))
    assert not out[0][:, mask.cuda() != 0].any()
    # the two layouts round in another order over a few steps
    assert _rel(out[0].double(), out[1].double()) < (1e-4 if precision == 4 else 1e-11)
