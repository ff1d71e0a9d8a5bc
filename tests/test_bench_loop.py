"""Which launches of a profiled step bench.py counts to the CG loop, for the
labels of a single grid and of a batch, after one and two iterations."""
import pytest

import bench

LOOP = {"sep_y": 2, "sep_x": 1, "sep_zi": 1, "sep_update": 1, "cg_dir_q": 1}   # launches per iteration
STEP = {"cfl_dt": 1, "advect_fused": 2, "momentum_fused": 1, "sep_init": 1, "project": 1, "turbulence": 1}


@pytest.mark.parametrize("prefix", ["", "b_"])
@pytest.mark.parametrize("iters", [1, 2, 3])
def test_separable_solve(prefix, iters):
    for k, per in LOOP.items():
        assert bench.loop_launches(prefix + k, per * iters, iters) == per, k
    for k, n in STEP.items():   # (a batch launches the advection once each for CFL and fixed time steps)
        assert bench.loop_launches(prefix + k, n, iters) == 0, k


@pytest.mark.parametrize("iters", [1, 2])
def test_batch_traffic(iters):
    kernels = {"b_" + k: dict(bytes_per_launch=10.0, launches=per * iters) for k, per in LOOP.items()}
    kernels.update({"b_" + k: dict(bytes_per_launch=100.0, launches=n) for k, n in STEP.items()})
    r = bench.step_traffic(kernels, iters, mean_iters=1.5, ms_per_step=1.0, peak=1.0, cells=1)
    assert r["per_cg_iteration_bytes_per_cell"] == 60.0 and r["fixed_bytes_per_cell"] == 700.0
    assert r["bytes"] == 700.0 + 1.5 * 60.0


def test_v_cycle_labels_keep_the_count():
    # seven iterations: once per iteration, and once more at the set-up
    assert bench.loop_launches("mg_up_L0", 8, 7) == 1 and bench.loop_launches("b_mg_tail", 8, 7) == 1
    assert bench.loop_launches("mg_up_L0", 0, 0) == 0


def test_the_solver_table_runs_what_its_rows_say():
    """The V-cycle of the default settings has to be asked for, or the separable inverse runs under its name."""
    rows = {name: (params, tuning) for name, params, tuning in bench.PRECONDITIONERS}
    assert len(rows) == len(bench.PRECONDITIONERS)
    default = [n for n, (p, _) in rows.items() if p.get("precond") == "mg" and p.get("mg_smoother", "cheby") == "cheby"
               and p.get("mg_transfer", "linear") == "linear"]
    assert sorted(default) == ["mg", "separable"]
    assert rows["mg"][1].get("coarse_start") == -1 and rows["separable"][1].get("coarse_start", 0) == 0


def test_the_mesh_roofline_counts_what_a_call_cannot_do_without():
    """5812 triangles on 256 x 256 x 64 in the 1.13 ms measured: 34 MB, far below the memory's rate, not above any peak."""
    r = bench.mesh_roofline(256 * 256 * 64, 5812, 1.13e-3, 6800.0, "measured")
    assert r["bound"] == "hbm" and abs(r["achieved"] - (72 * 5812 + 8 * 4194304) / 1.13e-3 / 1e9) < 1e-9
    assert 0.0 < r["frac"] < 0.01
