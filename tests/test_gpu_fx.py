"""FP64 right-hand sides at the edges of the fixed-point functions: grids and scales beyond their range (FP64
logarithms instead), the smallest tables, tables too large for shared memory, the flat regulator's kink, and
mass terms near the propagator pole; against the CPU oracle at the FP64 bar of the other tests."""
import dataclasses

import numpy as np
import pytest

import ffrg_inputs as fi
import oracle
from gpu_common import gpu_context

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gpu_context()
    yield c
    c.close()


def _grid(wl, lo, hi):
    wl.problem = dataclasses.replace(wl.problem, x_min=lo, x_max=hi, p_min=lo, p_max=hi)
    return wl


CASES = {
    "k above fixed point": lambda: (fi.make_d3(seed=1, n_ext_p=5, n_rad=16, n_ang=8), 3e9),
    "k below fixed point": lambda: (fi.make_d3(seed=2, n_ext_p=5, n_rad=16, n_ang=8), 2e-10),
    "grid below fixed point": lambda: (_grid(fi.make_d3(seed=3, n_ext_p=5, n_rad=16, n_ang=8), 1e-20, 10.0), 0.3),
    "two nodes": lambda: (fi.make_d3(seed=4, n_pts=2, n_ext_p=3, n_rad=9, n_ang=5), 1.0),
    "tables in global memory": lambda: (fi.make_d4(seed=5, n_pts=4000, n_ext_ang=1, n_rad=2, n_ang1=2, n_ang2=2), 1.0),
    "finite T tables in global memory": lambda: (fi.make_finite_t(seed=6, N=40, T=0.02, n_pts=160, n_ext_p=2, n_rad=8,
                                                                  n_ang=5), 0.7),
    "flat regulator": lambda: (fi.make_d3(seed=7, n_ext_p=9, n_rad=31, n_ang=11, regulator=fi.REG_LITIM), 1.0),
    "near the pole": lambda: (fi.make_d3(seed=8, n_ext_p=9, n_rad=16, n_ang=8, m2_over_k2=-0.97), 0.5),
    # the shape variables cancel the squares of legs 1e5 apart in length (an error of u p / q unless both sides
    # round the squares alike)
    "full vertex, small k": lambda: (fi.make_d4_full(seed=9, n_pts=12, n_va=3, n_vb=2, n_ext_ang=2, n_rad=8, n_ang1=6,
                                                     n_ang2=4), 1e-4),
}


@pytest.mark.parametrize("case", CASES)
def test_fp64_at_the_edges(ctx, case):
    import paper_2412_13043_gb300 as ffrg
    wl, k = CASES[case]()
    tabs = ctx.tables(wl.problem, wl.tables)
    got = ctx.rhs(wl.problem, tabs, k, precision=ffrg.FP64).cpu().numpy()
    tabs.free()
    ref = oracle.rhs(wl.problem, wl.tables, k)
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-12


@pytest.mark.parametrize("model,n_pts", [("d3", 20), ("d4", 12), ("d4", 37)])
def test_feedback_flow_does_not_depend_on_where_rows_are_computed(model, n_pts):
    """The FP64 RHS of feedback flows computes the rows of small problems in 32-row groups; without the row buffer
    (a context with a memory budget) each item's rows run in one warp.  Same bits either way."""
    import torch

    import paper_2412_13043_gb300 as ffrg
    if model == "d3":
        wl = fi.make_d3(seed=3, n_pts=n_pts, n_ext_p=n_pts, n_rad=37, n_ang=19, feedback=1, x_min=0.01)
    else:
        wl = fi.make_d4(seed=3, n_pts=n_pts, n_ext_ang=3, n_rad=21, n_ang1=13, n_ang2=5)
    ends = []
    for budget in (0, 1 << 30):
        c = ffrg.Context(0, hbm_budget_bytes=budget)
        tabs = c.tables(wl.problem, wl.tables)
        y = torch.tensor(wl.y0, dtype=torch.float64, device="cuda")
        c.flow(wl.problem, tabs, y, wl.Lambda, 2.0, feedback=1, rtol=1e-7)
        ends.append(y.cpu().numpy())
        c.close()
    assert np.array_equal(ends[0], ends[1])


@pytest.mark.parametrize("n_states", [1, 9, 257, 1025])
def test_states_do_not_depend_on_their_number(ctx, n_states):
    """The K ranges, and the blocks that share a state's slices, follow the number of states; the pass sums are
    integers and the scales per state: the same bits as one by one of the whole set, and the oracle's values."""
    import torch

    import paper_2412_13043_gb300 as ffrg
    wl = fi.make_finite_t(seed=11, N=15, T=0.01, n_pts=16, n_ext_p=5, n_ext_m=3, n_rad=133, n_ang=3)
    tabs = ctx.tables(wl.problem, wl.tables)
    rng = np.random.default_rng(12)
    F = rng.uniform(-1.0, 2.0, size=(1500, oracle.ft_nfreq(wl.problem), wl.problem.n_rad))
    dev = torch.from_numpy(F).cuda()
    whole = ctx.ft_states(wl.problem, tabs, 0.8, dev, precision=ffrg.FP64).cpu().numpy()
    some = ctx.ft_states(wl.problem, tabs, 0.8, dev[:n_states].contiguous(), precision=ffrg.FP64).cpu().numpy()
    tabs.free()
    assert np.array_equal(some, whole[:n_states])
    at = [0, n_states // 2, n_states - 1]
    ref = oracle.ft_states(wl.problem, wl.tables, 0.8, F[at])
    scale = oracle.ft_states(wl.problem, wl.tables, 0.8, np.abs(F[at]))
    assert np.max(np.abs(some[at] - ref) / scale) < 1e-12


@pytest.mark.parametrize("hi", [1.0 + 1e-9, 1.000001, 1.0001, 1.01])
@pytest.mark.parametrize("model", ["d3", "d4"])
def test_momenta_far_from_a_narrow_grid(ctx, model, hi):
    """Values and gradients on grids so narrow that a momentum lies up to 2^40 nodes outside: the end nodes."""
    import torch

    import paper_2412_13043_gb300 as ffrg
    wl = (fi.make_d3(seed=15, n_pts=64, n_ext_p=7, n_rad=16, n_ang=8) if model == "d3" else
          fi.make_d4(seed=15, n_pts=64, n_ext_ang=2, n_rad=5, n_ang1=3, n_ang2=3))
    wl.problem = dataclasses.replace(wl.problem, x_min=1.0, x_max=hi, p_min=0.01, p_max=3.0, n_ext_p=7)
    wl.tables = np.random.default_rng(16).uniform(0.5, 1.5, wl.tables.shape)
    gbar = np.random.default_rng(17).uniform(-1.0, 1.0, wl.problem.n_ext())
    tabs = ctx.tables(wl.problem, wl.tables)
    got = ctx.rhs(wl.problem, tabs, 0.3, precision=ffrg.FP64).cpu().numpy()
    grad = ctx.rhs_adjoint(wl.problem, tabs, 0.3, torch.tensor(gbar, device="cuda")).cpu().numpy().ravel()
    tabs.free()
    ref = oracle.rhs(wl.problem, wl.tables, 0.3)
    gref = oracle.rhs_jacobian(wl.problem, wl.tables, 0.3).T @ gbar
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-12
    assert np.max(np.abs(grad - gref)) / np.max(np.abs(gref)) < 1e-12


def _steep(wl):
    """Every momentum below the first node, the tables there 1e-12 of the next one."""
    wl.problem = dataclasses.replace(wl.problem, x_min=1.0, x_max=10.0, p_min=0.01, p_max=0.02, m2_over_k2=0.0,
                                     m2_shift=0.0)
    rng = np.random.default_rng(18)
    wl.tables = rng.uniform(0.5, 1.5, wl.tables.shape)
    wl.tables[..., 0] *= 1e-12
    return wl


STEEP = {
    "d3": lambda: fi.make_d3(seed=1, n_pts=12, n_ext_p=5, n_rad=9, n_ang=7),
    "d4": lambda: fi.make_d4(seed=1, n_pts=12, n_ext_ang=2, n_rad=7, n_ang1=5, n_ang2=3),
    "d4 full": lambda: fi.make_d4_full(seed=1, n_pts=12, n_va=3, n_vb=2, n_ext_ang=2, n_rad=7, n_ang1=5, n_ang2=3),
    "finite T": lambda: fi.make_finite_t(seed=1, N=4, T=1e-3, n_pts=12, n_ext_p=5, n_ext_m=2, n_rad=9, n_ang=7),
    "finite T, 4D regulator": lambda: fi.make_finite_t_4d(seed=1, N=8, T=1e-3, n_pts=12, n_ext_p=5, n_ext_m=2, n_rad=9,
                                                          n_ang=7, n_x0=9),
    "tables in global memory": lambda: fi.make_d4(seed=1, n_pts=4000, n_ext_ang=1, n_rad=3, n_ang1=2, n_ang2=2),
    "grid beyond fixed point": lambda: fi.make_d3(seed=1, n_pts=12, n_ext_p=5, n_rad=9, n_ang=7),
}


@pytest.mark.parametrize("case", STEEP)
def test_lookups_below_a_steep_first_cell(ctx, case):
    """Below the grid a table has its first value, however far the second is from it."""
    import torch

    import paper_2412_13043_gb300 as ffrg
    wl = _steep(STEEP[case]())
    wl.problem = dataclasses.replace(wl.problem, n_ext_p=5, x_max=1e17 if case == "grid beyond fixed point" else 10.0)
    tabs = ctx.tables(wl.problem, wl.tables)
    got = ctx.rhs(wl.problem, tabs, 0.01, precision=ffrg.FP64).cpu().numpy()
    ref = oracle.rhs(wl.problem, wl.tables, 0.01)
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-12
    if case in ("d3", "d4", "grid beyond fixed point"):
        gbar = np.random.default_rng(19).uniform(0.5, 1.0, wl.problem.n_ext())
        grad = ctx.rhs_adjoint(wl.problem, tabs, 0.01, torch.tensor(gbar, device="cuda")).cpu().numpy().ravel()
        gref = oracle.rhs_jacobian(wl.problem, wl.tables, 0.01).T @ gbar
        assert np.max(np.abs(grad - gref)) / np.max(np.abs(gref)) < 1e-12
    tabs.free()


@pytest.mark.parametrize("case", ["d4", "finite T", "d4, below the grid", "finite T, below the grid"])
def test_large_tables_in_a_context_with_a_tight_budget(case):
    """Tables beyond shared memory need no more device memory than themselves, their FP32 copy and a plan's small
    buffers: read in place, without the line form (192 KB and 251 KB here) that a context without a budget keeps."""
    import paper_2412_13043_gb300 as ffrg
    if case.startswith("d4"):
        wl = fi.make_d4(seed=5, n_pts=4000, n_ext_ang=1, n_rad=5, n_ang1=4, n_ang2=3)
    else:
        wl = fi.make_finite_t(seed=6, N=40, T=0.02, n_pts=160, n_ext_p=2, n_rad=8, n_ang=5)
    k = 0.7
    if case.endswith("grid"):
        wl, k = _steep(wl), 0.01
        wl.problem = dataclasses.replace(wl.problem, T=1e-4)
    wl.problem = dataclasses.replace(wl.problem, n_ext_p=5)
    c = ffrg.Context(0, hbm_budget_bytes=2 * wl.tables.nbytes + (64 << 10))
    tabs = c.tables(wl.problem, wl.tables)
    ref = oracle.rhs(wl.problem, wl.tables, k)
    for precision, tol in ((ffrg.FP64, 1e-12),) + (((ffrg.MIXED, 1e-6),) if case in ("d4", "finite T") else ()):
        got = c.rhs(wl.problem, tabs, k, precision=precision).cpu().numpy()
        assert np.max(np.abs(got - ref) / np.abs(ref)) < tol
    c.close()
