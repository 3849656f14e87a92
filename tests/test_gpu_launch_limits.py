"""Launches whose shared memory lies at the limit a kernel gets unasked (48 KB, static and
dynamic together), in a process that has launched nothing larger before."""
import os
import subprocess
import sys

import numpy as np
import pytest

from synth import NetSpec, Problem, init_params, make_batch
from synth.workloads import PDE_BURGERS, PDE_NS

from gpu_helpers import TOL, assert_parity, run_oracle

pytestmark = pytest.mark.gpu

# The output kernel holds 76 bytes of dynamic shared memory per unit of the last layer with
# three outputs and 36 with one: these widths end just below 48 KB of it.
WIDTHS = [(PDE_NS, 586), (PDE_NS, 646), (PDE_BURGERS, 1237), (PDE_BURGERS, 1365)]
PROBLEM = Problem(0.02, 0.3, 2.0, 5.0)


def _inputs(pde, width):
    spec = NetSpec(pde, 2, 3 if pde == PDE_NS else 1, [16, width], rwf=True)
    return spec, init_params(spec, 41, 0.2), make_batch(pde, 200, 0 if pde == PDE_NS else 20, 30, 42, 43)


def _run(out):
    from gpu_helpers import run_gpu
    res = {}
    for pde, width in WIDTHS:
        spec, p, b = _inputs(pde, width)
        for precision in ("fp32", "bf16"):
            t, g = run_gpu(spec, p, None, b, PROBLEM, precision)
            res[f"t_{pde}_{width}_{precision}"], res[f"g_{pde}_{width}_{precision}"] = t, g
    np.savez(out, **res)


def test_output_kernel_just_below_the_default_limit(cuda_lib, tmp_path):
    out = str(tmp_path / "res.npz")
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(here), here, os.environ.get("PYTHONPATH", "")]))
    r = subprocess.run([sys.executable, os.path.abspath(__file__), out], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    res = np.load(out)
    for pde, width in WIDTHS:
        spec, p, b = _inputs(pde, width)
        rt, rg = run_oracle(spec, p, None, b, PROBLEM)
        assert_parity(res[f"t_{pde}_{width}_fp32"], res[f"g_{pde}_{width}_fp32"], rt, rg, TOL["fp32"],
                      f"last layer {width}", spec=spec)
        # BF16: the total and the whole gradient (a residual of a few points may cancel below its tolerance)
        t, g = res[f"t_{pde}_{width}_bf16"], res[f"g_{pde}_{width}_bf16"]
        assert abs(t[0] - rt[0]) <= TOL["bf16"] * abs(rt[0])
        assert np.linalg.norm(g - rg) <= TOL["bf16"] * np.linalg.norm(rg)


if __name__ == "__main__":
    _run(sys.argv[1])
