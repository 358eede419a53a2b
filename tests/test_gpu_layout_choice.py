"""The automatic layout of D2Q9 solvers against calls that change it or its kernels."""
import time

import numpy as np
import pytest
import torch

from paper_2310_00810_gb300 import autotune
from paper_2310_00810_gb300 import lbm
from paper_2310_00810_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def dev(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x)).to(device="cuda", dtype=dtype)


def _mask(nx, ny, seed=2, solid=0.2):
    m = (np.random.Generator(np.random.PCG64(seed)).uniform(size=(ny, nx)) < solid).astype(np.uint8)
    m[:, :2] = m[:, -2:] = 0
    return torch.as_tensor(m)


def _solver(nx=64, ny=40, T=30, layout=None, precision=4, **kw):
    return lbm.Solver(9, nx, ny, precision=precision, n_steps=T, inlet_kind=lbm.LBM_INLET_PROFILE,
                      geometry=_mask(nx, ny), layout=layout, **kw)


def _inputs(s, seed=5):
    return (dev(1.0 + W.inlet_profile(s.plan.n_in, seed=seed)), dev([0.73]), 1.0), \
        dev(W.perturbation((2, *s.plan.shape), seed=seed + 1, scale=1e-4))


def _gradient(s, between=lambda s: None):
    p, ut = _inputs(s)
    f = s.forward(*p)
    loss, lam = s.loss_grad(f, ut)
    between(s)
    return (f, loss, lam, *s.adjoint(*p, lam))


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


# calls that left a default solver's checkpoints alone while its layout was the dense one
BETWEEN = {
    "family": lambda s: s.set_kernels(step_family=lbm.LBM_FAMILY_VEC, adjoint_family=lbm.LBM_FAMILY_VEC),
    "dense": lambda s: s.set_layout("dense"),
    "two_steps": lambda s: s.set_kernels(steps_per_launch=2),
    "family_then_step": lambda s: (s.set_kernels(step_family=lbm.LBM_FAMILY_VEC), s.step(*_inputs(s)[0], s.new_state().zero_(), 3)),
}


@pytest.mark.parametrize("precision", [4, 8])
@pytest.mark.parametrize("between", list(BETWEEN))
def test_a_layout_named_between_the_sweeps_takes_effect_at_the_next_forward(between, precision):
    s = _solver(precision=precision)
    want = _gradient(s)
    got = _gradient(s, BETWEEN[between])
    assert torch.count_nonzero(want[3]).item() > 0
    assert _same(got, want)
    assert s.layout == "dense"
    f = s.forward(*_inputs(s)[0])
    assert s.layout == "dense" and s.tables is None
    assert torch.allclose(f, want[0], rtol=0.0, atol=1e-6 if precision == 4 else 1e-13)


@pytest.mark.parametrize("q,first,second", [(9, "compact", "dense"), (9, "dense", "compact"), (19, "compact", "dense")])
def test_a_reverse_sweep_after_a_change_of_layout_is_refused(q, first, second):
    if q == 9:
        s = _solver(layout=first)
    else:
        s = lbm.Solver(19, 20, 12, 9, n_steps=10, inlet_kind=lbm.LBM_INLET_PROFILE, layout=first)
    p = (dev(1.0 + W.inlet_profile(s.plan.n_in, seed=5)), dev([0.8]), 1.0)
    f = s.forward(*p)
    _, lam = s.loss_grad(f, dev(W.perturbation((s.plan.d, *s.plan.shape), seed=6, scale=1e-4)))
    s.set_layout(second)
    with pytest.raises(lbm.LBMError) as e:
        s.adjoint(*p, lam)
    assert e.value.status == lbm.LBM_ERR_INVALID_ARG
    s.forward(*p)
    g_in, _ = s.adjoint(*p, lam)
    assert torch.count_nonzero(g_in).item() > 0


@pytest.mark.parametrize("choice", [dict(step_family=lbm.LBM_FAMILY_VEC), dict(persist=1), dict(pdl=0)])
def test_kernels_after_a_velocity_inlet(choice):
    """The inlet runs in the fluid-only layout, rounding as that layout named does, whatever is named later."""
    out = []
    for layout, kernels in ((None, None), (None, choice), ("compact", None)):
        s = _solver(layout=layout)
        s.set_velocity_inlet((0.05, 0.0))
        if kernels:
            s.set_kernels(**kernels)
        assert s.layout == "compact"
        out.append(_gradient(s))
    assert _same(out[0], out[1]) and _same(out[0], out[2])


def test_another_geometry_moves_the_solver_to_the_dense_layout():
    s = _solver()
    m = _mask(64, 40, seed=9).cuda()
    s.mask[: s.plan.N].copy_(m.reshape(-1))
    lbm.lbm_init_geometry(s.plan, s.mask, s.link, s.info, s.porosity, kind=lbm.LBM_GEOM_MASK, fill_isolated=False)
    # the plan is dense from here on; a sweep through s.ws must find room for it
    assert s.layout == "dense"
    assert s.ws.numel() >= lbm.lbm_workspace_size(s.plan)
    fresh = lbm.Solver(9, 64, 40, n_steps=30, inlet_kind=lbm.LBM_INLET_PROFILE, geometry=m, layout="dense")
    assert _same(_gradient(s), _gradient(fresh))
    s.set_velocity_inlet((0.05, 0.0))
    assert s.layout == "compact"
    assert torch.isfinite(s.forward(*_inputs(s)[0])).all()


@pytest.mark.parametrize("first", ["aa", "extrap"])
def test_in_place_streaming_on_the_automatic_layout(first):
    """It is ignored there, as it was while the dense layout was the automatic one."""
    want = _solver()
    lbm.lbm_set_abb_velocity(want.plan, lbm.LBM_ABB_U_EXTRAP)
    s = _solver()
    for name in ("aa", "extrap") if first == "aa" else ("extrap", "aa"):
        if name == "aa":
            s.set_kernels(aa=1)
        else:
            s.set_abb_velocity(lbm.LBM_ABB_U_EXTRAP)
    assert _same(_gradient(s), _gradient(want))
    s = _solver()
    want = _gradient(s)
    assert _same(_gradient(s, lambda s: s.set_kernels(aa=1)), want)


def test_only_another_dense_choice_leaves_the_automatic_layout():
    s = _solver()
    for choice in (dict(persist=0), dict(vec=4, tma_rows=8), dict(steps_per_launch=1), dict(adjoint_tma_rows=0),
                   dict(step_family=lbm.LBM_FAMILY_AUTO, pdl=0), lbm.lbm_plan_get_kernels(s.plan)):
        s.set_kernels(**choice)
        assert s.layout == "compact", choice
    s.set_kernels(recompute_family=lbm.LBM_FAMILY_VEC)
    assert s.layout == "dense"


# rows that the one-node-per-thread kernels take where the TMA or register kernels apply too
@pytest.mark.parametrize("nx,ny", [(64, 40), (66, 40), (512, 128)])
def test_the_dense_layouts_kernel_families_round_alike(nx, ny):
    out = []
    for family in (lbm.LBM_FAMILY_AUTO, lbm.LBM_FAMILY_VEC):
        s = _solver(nx, ny, layout="dense")
        lbm.lbm_plan_set_kernels(s.plan, step_family=family, adjoint_family=family)
        out.append(_gradient(s))
    (f, _, lam, g_in, g_tau), (fv, _, lamv, gv, tv) = out
    assert torch.equal(f, fv) and torch.equal(lam, lamv)
    # FP32 adjoint states of other compilations, FP32 warp sums over other groups of nodes
    assert ((g_in - gv).norm() / gv.norm()).item() < 1e-6 and abs((g_tau - tv) / tv).item() < 1e-5


# tau = 0.73: 1 / tau rounded from FP64 and the quotient of the FP32 numbers differ
@pytest.mark.parametrize("nx", [64, 65])
def test_tuning_keeps_the_rounding_of_the_automatic_layout(nx):
    s = _solver(nx, 41)
    before = _gradient(s)
    autotune._apply(s, dict(layout="compact", choice=dict(pdl=1, overlap=0, aa=1)))
    assert s.layout == "compact" and lbm.lbm_plan_get_kernels(s.plan)["aa"] == 1
    assert _same(_gradient(s), before)


def test_tuning_results_are_kept_apart_by_what_decides_them(tmp_path):
    cache = str(tmp_path / "t.json")
    s = _solver(65, 41)
    autotune.tune(s, t_tune=8, repeats=1, cache=cache)
    assert autotune.tune(s, t_tune=8, repeats=1, cache=cache)["cached"]
    mrt = _solver(65, 41)
    mrt.set_collision(lbm.LBM_COLLISION_MRT, 1.1, 1.1, 1.2)
    assert not autotune.tune(mrt, t_tune=8, repeats=1, cache=cache)["cached"]
    opened = lbm.Solver(9, 65, 41, n_steps=30, inlet_kind=lbm.LBM_INLET_PROFILE, geometry=_mask(65, 41, solid=0.0))
    assert not autotune.tune(opened, t_tune=8, repeats=1, cache=cache)["cached"]


@pytest.mark.parametrize("layout", ["dense", "compact"])
def test_naming_the_layout_it_has_keeps_the_captured_sweeps(layout):
    """A sweep after it costs the host a replay, not a capture of thousands of launches (milliseconds)."""
    s = _solver(T=6000, layout=layout)
    p, _ = _inputs(s)
    f = s.new_state()

    def host_ms():
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s.forward(*p, f)
        dt = (time.perf_counter() - t0) * 1e3
        torch.cuda.synchronize()
        return dt

    def again():
        s.set_layout(layout)
        return host_ms()

    first = host_ms()
    same = min(host_ms() for _ in range(3))
    assert first > 2.0
    assert min(again() for _ in range(3)) < max(5 * same, 1.5)


def test_a_refused_choice_changes_nothing():
    s = _solver()
    want = _gradient(s)
    with pytest.raises(ValueError):
        s.set_layout("sparse")
    with pytest.raises(lbm.LBMError):
        s.set_kernels(step_family=9)
    assert s.layout == "compact" and _same(_gradient(s), want)
    s.set_kernels(step_family=lbm.LBM_FAMILY_VEC)  # the layout is still automatic
    s.forward(*_inputs(s)[0])
    assert s.layout == "dense"
