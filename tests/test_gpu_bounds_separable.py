"""The bounds-checked build over the separable inverse and the kernels that
walk their arrays by pointer, at the shapes that take another path through them:
folded and unfolded axes, one cell in z, narrow panels, odd sizes, a batch."""
import os
import re
import subprocess
import sys
import textwrap

import pytest

from paper_2204_01117_gb300 import uf

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = textwrap.dedent("""
    import os, sys
    import numpy as np
    sys.path.insert(0, os.environ["UF_ROOT"])
    from paper_2204_01117_gb300 import uf
    assert uf.load().uf_bounds_checked() == 1
    def city(g, seed):
        phi = np.where(np.random.default_rng(seed).random(g.shapes["phi"]) < 0.1, 0.0, 1.0)
        g.set_porosity(phi.astype(g.np_dtype))
        g.init_state()
    for precision in ("f32", "f64"):
        for (dims, deg) in (((33, 45, 9), 0.0), ((48, 40, 16), 180.0), ((70, 37, 21), 90.0), ((57, 31, 12), 230.0), ((64, 70, 1), 0.0),
                            ((40, 36, 1), 45.0), ((2, 2, 2), 0.0), ((129, 20, 5), 270.0), ((24, 769 if precision == "f32" else 301, 2), 0.0)):
            g = uf.Grid(*dims, precision=precision, wind_dir_deg=deg)
            assert g.get_tuning()[0]["coarse_start"] == 0
            city(g, dims[0])
            g.run(2)
            g.close()
    bt = uf.Batch([dict(nx=n, ny=m, nz=k, wind_dir_deg=d, **kw) for n, m, k, d, kw in
                   ((48, 40, 16, 0.0, {}), (35, 29, 11, 120.0, {}), (40, 33, 1, 90.0, {}), (31, 24, 9, 0.0, dict(fixed_dt=0.1)))])
    for i, g in enumerate(bt.grids):
        city(g, i)
    bt.run(2)
    bt.close()
    print("clean")
""")


@pytest.mark.gpu
def test_bounds_checked_build_runs_them_clean():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    env = dict(os.environ, UF_LIBRARY=uf.build(checked=True), UF_ROOT=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=1500)
    assert r.returncode == 0 and "clean" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def body(header, name):
    """Source of function `name`, comments left out."""
    with open(os.path.join(ROOT, "paper_2204_01117_gb300", "csrc", header)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = text.index("{", text.index(" " + name + "("))
    depth = 0
    for at in range(start, len(text)):
        depth += (text[at] == "{") - (text[at] == "}")
        if depth == 0:
            return text[start:at + 1]


WALKERS = {"sep_solve.cuh": {"sep_zf": ("S.t",), "sep_apply": ("f",), "sep_init_body": ("b", "x", "L.r"),
                             "sep_update_body": ("L.r", "q", "dn", "x"), "sep_zi_body": ("S.t",), "sep_y_panel": ("src",)},
           "mg_fused.cuh": {"cg_dir_q_body": ("z", "dold", "dnew", "q")},
           "solver_kernels.cuh": {"cg_init_body": ("gp",)},
           "step_kernels.cuh": {"turbulence_body": ("pu", "pv", "pw"), "project_cells_body": ("pu", "pv", "pw", "pc")},
           "advect_fused.cuh": {"stage_plane": ("su", "sv", "sw")},
           "momentum_fused.cuh": {"stage_momentum": ("su", "sv", "sw", "sn", "sc"), "u3_plane": ("gu", "gv", "gw")}}


@pytest.mark.parametrize("header, name", [(h, n) for h, fs in WALKERS.items() for n in fs])
def test_walking_kernels_pass_their_pointers_through_the_check(header, name):
    src = body(header, name)
    for ptr in WALKERS[header][name]:
        p = re.escape(ptr)
        # no direct access: ptr[..], *(ptr ..), a vector read or write at ptr, an asynchronous copy from it
        for direct in (rf"(?<![\w.]){p}\[", rf"\*\({p} ", rf"reinterpret_cast<[^>]*>\({p}\b", rf"cp_async_elem\([^;]*, {p} "):
            assert not re.search(direct, src), (ptr, direct, re.search(direct, src).group(0))
