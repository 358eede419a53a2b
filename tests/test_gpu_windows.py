"""The fluid-only kernels' neighbour search (windows of 30 columns, boundary columns through the table) and
their launch forms, against the CPU oracle at the sizes where each can go wrong: row lengths around the
window's edges, columns next to the boundary columns, lattices too narrow for windows, periodic rows, rows
of solid nodes, and node counts on both sides of the pipelined kernels' threshold."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2310_00810_gb300 import lbm
from paper_2310_00810_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# FP64: both sides round each operation to 1 ulp in another order, over a few steps; FP32 as the parity tests
TOL = {8: (1e-11, 1e-9), 4: (1e-4, 1e-3)}


def dev(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x)).to(device="cuda", dtype=dtype)


def rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(np.asarray(b)), 1e-300)


def _mask(shape, seed, solid=0.25):
    m = (np.random.Generator(np.random.PCG64(seed)).uniform(size=shape) < solid).astype(np.uint8)
    m[..., shape[-2] // 2, :] = 1  # a row of solid nodes
    m[..., 0, :2] = 0
    return m


def _check(q, m, precision, T, periodic=False, seed=1):
    shape = m.shape
    nx, ny, nz = shape[-1], shape[-2], shape[0] if q == 19 else 1
    s = lbm.Solver(q, nx, ny, nz, precision=precision, n_steps=T, inlet_kind=lbm.LBM_INLET_PROFILE,
                   geometry=torch.as_tensor(m), layout="compact", periodic_y=periodic)
    rin = 1.0 + W.inlet_profile(ny * nz, seed=seed)
    ut = W.perturbation((s.plan.d, *shape), seed=seed + 1, scale=1e-3)
    _, w, _ = O.lattice(q)
    f0 = W.perturbation((q, *shape), seed=seed + 2, scale=2e-3)
    f0[:, m == 1] = 0.0
    wb = w.reshape(-1, *([1] * len(shape)))
    with O.wake_options(periodic_y=periodic):
        want = O.forward(q, m, rin, 1.0, 0.8, 3, f0=f0 + wb) - wb
        Lw, gw, gtw = O.gradient(q, m, rin, 1.0, 0.8, T, ut, ckpt_stride=s.plan.desc.ckpt_stride or 0)[:3]
    got = s.step(dev(rin), dev([0.8]), 1.0, dev(f0, s.plan.dtype), 3).cpu().numpy()
    fl = m == 0
    tol_f, tol_g = TOL[precision]
    assert rel(got[:, fl], want[:, fl]) < tol_f
    f = s.forward(dev(rin), dev([0.8]), 1.0)
    L, lam = s.loss_grad(f, dev(ut))
    g_in, g_tau = s.adjoint(dev(rin), dev([0.8]), 1.0, lam)
    assert abs(L.item() - Lw) <= tol_f * abs(Lw)
    assert rel(g_in.cpu().numpy(), gw) < tol_g
    assert abs(g_tau.item() - gtw) <= tol_g * abs(gtw)


@pytest.mark.parametrize("nx", [2, 3, 4, 5, 29, 30, 31, 32, 33, 59, 60, 61, 62, 91])
@pytest.mark.parametrize("periodic", [False, True])
def test_row_lengths_2d(nx, periodic):
    _check(9, _mask((7, nx), 10 + nx), 8, 7, periodic, seed=nx)


@pytest.mark.parametrize("nx", [3, 4, 30, 32, 61])
def test_row_lengths_3d(nx):
    _check(19, _mask((5, 6, nx), 20 + nx), 8, 5, seed=nx)


@pytest.mark.parametrize("ny", [1, 2, 3])
def test_few_rows(ny):
    m = np.zeros((ny, 40), np.uint8)
    m[ny // 2, 11:13] = 1 if ny > 1 else 0
    _check(9, m, 8, 6, seed=ny)


# just below and above 600000 fluid nodes, and several times that: simple and pipelined launches, D2Q9 FP32
@pytest.mark.parametrize("nx,ny", [(1000, 790), (1000, 810), (1511, 1301)])
def test_pipelined_and_simple_launches(nx, ny):
    m = (np.random.Generator(np.random.PCG64(3)).uniform(size=(ny, nx)) < 0.25).astype(np.uint8)
    _check(9, m, 4, 4)


def test_batch_takes_both_node_block_classes():
    """A batch past the pipelined kernels' threshold gives bit for bit the states and gradients of single plans
    of the same launches: its blocks of interior nodes alone and those with boundary or padding nodes."""
    sizes = [(1024, 512, 1), (992, 480, 1), (64, 32, 1), (1024, 500, 1)]
    geoms = [dict(kind=lbm.LBM_GEOM_DISKS, seed=50 + i, r_min=3, r_max=6, target_porosity=0.7) for i in range(4)]
    T = 6
    b = lbm.Batch(9, sizes, precision=4, n_steps=T, inlet_kind=lbm.LBM_INLET_PROFILE, geometries=geoms,
                  layout="compact")
    rho = b.new_inlet()
    ut = b.new_velocity()
    for i, (nx, ny, _) in enumerate(sizes):
        b.view_inlet(rho, i).copy_(dev(1.0 + W.inlet_profile(ny, seed=60 + i)))
        b.view_velocity(ut, i).copy_(dev(W.perturbation((2, ny, nx), seed=70 + i, scale=1e-3)))
    tau = dev([0.8, 0.75, 0.9, 1.0])
    f = b.forward(rho, tau, 1.0)
    _, lam = b.loss_grad(f, ut)
    g_in, g_tau = b.adjoint(rho, tau, 1.0, lam)
    for i, (nx, ny, _) in enumerate(sizes):
        s = lbm.Solver(9, nx, ny, precision=4, n_steps=T, inlet_kind=lbm.LBM_INLET_PROFILE, geometry=geoms[i],
                       layout="compact")
        r, t = b.view_inlet(rho, i).clone(), tau[i:i + 1].clone()
        assert torch.equal(s.forward(r, t, 1.0), b.view_state(f, i))
        gi, gt = s.adjoint(r, t, 1.0, b.view_state(lam, i).contiguous())
        assert torch.equal(gi, b.view_inlet(g_in, i)) and torch.equal(gt, g_tau[i:i + 1])


# rows of 4 k and of 4 k + 2 nodes: the dense layout's TMA and register kernels
@pytest.mark.parametrize("nx,ny", [(64, 40), (66, 40), (512, 128)])
def test_the_automatic_layout_rounds_as_the_dense_one(nx, ny):
    m = (np.random.Generator(np.random.PCG64(nx)).uniform(size=(ny, nx)) < 0.2).astype(np.uint8)
    T, rin, ut = 30, dev(1.0 + W.inlet_profile(ny, seed=5)), dev(W.perturbation((2, ny, nx), seed=6, scale=1e-4))
    out = []
    for layout in (None, "dense"):
        s = lbm.Solver(9, nx, ny, precision=4, n_steps=T, inlet_kind=lbm.LBM_INLET_PROFILE,
                       geometry=torch.as_tensor(m), layout=layout)
        if layout:
            lbm.lbm_plan_set_kernels(s.plan, step_family=lbm.LBM_FAMILY_VEC, adjoint_family=lbm.LBM_FAMILY_VEC)
        else:
            assert s.layout == "compact"
        f = s.forward(rin, dev([0.8]), 1.0)
        _, lam = s.loss_grad(f, ut)
        out.append((f, lam, *s.adjoint(rin, dev([0.8]), 1.0, lam)))
    (f, lam, g_in, g_tau), (fd, lamd, gd, td) = out
    assert torch.equal(f, fd) and torch.equal(lam, lamd)
    assert rel(g_in.cpu().numpy(), gd.cpu().numpy()) < 1e-6  # FP32 adjoint states, other compilations
    assert rel(g_tau.cpu().numpy(), td.cpu().numpy()) < 1e-5  # FP32 warp sums over other groups of nodes
    s = lbm.Solver(9, nx, ny, precision=4, n_steps=T, geometry=torch.as_tensor(m))
    s.set_kernels(step_family=lbm.LBM_FAMILY_VEC)
    assert s.layout == "dense"


# odd rows, and options without a vector or TMA kernel: the dense layout's one-node-per-thread kernels.  tau = 0.73:
# 1 / tau rounded from FP64 and the quotient of the FP32 numbers differ.
@pytest.mark.parametrize("nx,ny,option", [(65, 40, None), (301, 149, None), (64, 40, "mrt"), (64, 40, "extrap")])
def test_the_automatic_layout_is_as_accurate_as_one_node_per_thread(nx, ny, option):
    m = (np.random.Generator(np.random.PCG64(nx)).uniform(size=(ny, nx)) < 0.2).astype(np.uint8)
    T, rin, ut = 30, dev(1.0 + W.inlet_profile(ny, seed=5)), dev(W.perturbation((2, ny, nx), seed=6, scale=1e-4))
    out = []
    for layout in (None, "dense"):
        s = lbm.Solver(9, nx, ny, precision=4, n_steps=T, inlet_kind=lbm.LBM_INLET_PROFILE,
                       geometry=torch.as_tensor(m), layout=layout)
        if option == "mrt":
            s.set_collision(lbm.LBM_COLLISION_MRT, 1.1, 1.1, 1.2)
        elif option == "extrap":
            lbm.lbm_set_abb_velocity(s.plan, lbm.LBM_ABB_U_EXTRAP)
        f = s.forward(rin, dev([0.73]), 1.0)
        _, lam = s.loss_grad(f, ut)
        out.append((f, *s.adjoint(rin, dev([0.73]), 1.0, lam)))
    (f, g_in, g_tau), (fd, gd, td) = out
    assert torch.allclose(f, fd, rtol=0.0, atol=4e-7 * float(fd.abs().max()))  # T steps of contraction differences
    assert rel(g_in.cpu().numpy(), gd.cpu().numpy()) < 1e-5
    assert rel(g_tau.cpu().numpy(), td.cpu().numpy()) < 1e-5


def _default_and_dense(nx, ny, option, T=5):
    """(state, seed, dL/drho_in, dL/dtau) of the automatic layout and of the dense layout's register (even rows)
    or one-node-per-thread kernels (odd rows, or an option that only they have)."""
    m = (np.random.Generator(np.random.PCG64(nx)).uniform(size=(ny, nx)) < 0.25).astype(np.uint8)
    rin, ut = dev(1.0 + W.inlet_profile(ny, seed=5)), dev(W.perturbation((2, ny, nx), seed=6, scale=1e-4))
    out = []
    for layout in (None, "dense"):
        s = lbm.Solver(9, nx, ny, precision=4, n_steps=T, inlet_kind=lbm.LBM_INLET_PROFILE,
                       geometry=torch.as_tensor(m), layout=layout)
        assert int(s.info[3].item()) > 600000
        if option == "mrt":
            s.set_collision(lbm.LBM_COLLISION_MRT, 1.1, 1.1, 1.2)
        elif option == "extrap":
            s.set_abb_velocity(lbm.LBM_ABB_U_EXTRAP)
        if layout:
            family = lbm.LBM_FAMILY_VEC if nx % 2 == 0 else lbm.LBM_FAMILY_SCALAR
            lbm.lbm_plan_set_kernels(s.plan, step_family=family, adjoint_family=family)
        else:
            assert s.layout == "compact"
        f = s.forward(rin, dev([0.73]), 1.0)
        _, lam = s.loss_grad(f, ut)
        out.append((f, lam, *s.adjoint(rin, dev([0.73]), 1.0, lam)))
    return out


# past the pipelined kernels' threshold, in the rounding of the automatic layout
@pytest.mark.parametrize("nx,ny,option", [(1000, 830, None), (1001, 831, None), (1000, 830, "mrt"),
                                          (1001, 831, "mrt"), (1000, 830, "extrap"), (1001, 831, "extrap")])
def test_the_automatic_layout_past_the_pipelined_threshold(nx, ny, option):
    (f, lam, g_in, g_tau), (fd, lamd, gd, td) = _default_and_dense(nx, ny, option)
    if option is None and nx % 2 == 0:
        assert torch.equal(f, fd) and torch.equal(lam, lamd)
    else:
        assert torch.allclose(f, fd, rtol=0.0, atol=4e-7 * float(fd.abs().max()))  # contraction differences
    assert rel(g_in.cpu().numpy(), gd.cpu().numpy()) < 1e-5
    assert rel(g_tau.cpu().numpy(), td.cpu().numpy()) < 1e-5


@pytest.mark.parametrize("mrt", [False, True])
def test_a_periodic_lattice_repeated_past_the_pipelined_threshold(mrt):
    """A lattice periodic in y with a ramped velocity inlet, and nine copies of it one above the other: the same
    flow, by one node per thread and by the pipelined kernels."""
    nx, ny, copies, T = 1000, 90, 9, 6
    m = (np.random.Generator(np.random.PCG64(8)).uniform(size=(ny, nx)) < 0.2).astype(np.uint8)
    ut = W.perturbation((2, 2, ny, nx), seed=9, scale=1e-3)
    out = []
    for n in (1, copies):
        s = lbm.Solver(9, nx, n * ny, precision=4, n_steps=T, geometry=torch.as_tensor(np.tile(m, (n, 1))),
                       periodic_y=True)
        assert (int(s.info[3].item()) > 600000) == (n == copies)
        s.set_velocity_inlet((0.05, 0.01))
        s.set_velocity_ramp(4)
        if mrt:
            s.set_collision(lbm.LBM_COLLISION_MRT, 1.1, 1.1, 1.2)
        f = s.forward(dev([1.0]), dev([0.73]), 1.0)
        L, _, g = s.adjoint_window(dev([1.0]), dev([0.73]), 1.0, f, [3, T], dev(np.tile(ut, (1, 1, n, 1))))
        out.append((f.cpu().numpy(), L.item(), g.item()))
    (f1, L1, g1), (fn, Ln, gn) = out
    # the same operations per node, of two compilations
    assert np.abs(fn - np.tile(f1, (1, copies, 1))).max() <= 4e-7 * np.abs(f1).max()
    assert abs(Ln - copies * L1) <= 1e-5 * abs(Ln) and abs(gn - copies * g1) <= 1e-4 * abs(gn)
