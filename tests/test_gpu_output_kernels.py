"""The three output/loss kernels against the FP64 oracle, BF16 (their only precision
for the first two):

* width <= 256, a multiple of 32: the output layer's contractions on warp-level
  tensor-core MMAs (k_out_loss_mma), for one output (Burgers jet rule) and three
  (Navier-Stokes and Maxwell jet rules), with initial and boundary sets and masks;
* width <= 512, a multiple of 32: the CUDA-core kernel fed by the same TMA ring
  (k_out_loss_tma);
* any other width: the register-tiled kernel (k_out_loss).
Each case runs a few hundred points over several tiles and a ragged tail, so every
consumer warp of the TMA kernels sees interior, initial, boundary and padding points."""
import dataclasses

import pytest

from synth import NetSpec, Problem, init_params, ff_matrix, make_batch
from synth.workloads import PDE_BURGERS, PDE_NS, PDE_MAXWELL, PDE_ALLEN_CAHN

from gpu_helpers import TOL, assert_parity, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def _case(pde, d_in, d_out, widths, ff, n_res, n_ic, n_bc, seed, masks=None):
    spec = NetSpec(pde, d_in, d_out, widths, ff_m=ff, ff_sigma=1.0, rwf=True)
    p = init_params(spec, seed, 0.15)
    B = ff_matrix(spec, seed + 1) if ff else None
    b = make_batch(pde, n_res, n_ic, n_bc, seed + 2, seed + 3)
    if masks is not None:
        b = dataclasses.replace(b, ic_mask=masks[0], bc_mask=masks[1])
    return spec, p, B, b


@pytest.mark.parametrize("widths", [[64, 32], [96, 128], [64, 256]])
def test_mma_output_kernel_navier_stokes(cuda_lib, widths):
    spec, p, B, b = _case(PDE_NS, 2, 3, widths, 16, 700, 0, 190, 301)
    gt, gg = run_gpu(spec, p, B, b, Problem(0.02, 0.7, 1.0, 3.0), "bf16")
    rt, rg = run_oracle(spec, p, B, b, Problem(0.02, 0.7, 1.0, 3.0))
    assert_parity(gt, gg, rt, rg, TOL["bf16"], f"NS {widths}", spec=spec)


@pytest.mark.parametrize("widths,masks", [([128, 128, 128], None), ([64, 160], (0b110, 0b011))])
def test_mma_output_kernel_maxwell(cuda_lib, widths, masks):
    spec, p, B, b = _case(PDE_MAXWELL, 3, 3, widths, 0, 500, 120, 150, 311, masks)
    gt, gg = run_gpu(spec, p, B, b, Problem(0.0, 1.0, 2.0, 0.5), "bf16")
    rt, rg = run_oracle(spec, p, B, b, Problem(0.0, 1.0, 2.0, 0.5))
    assert_parity(gt, gg, rt, rg, TOL["bf16"], f"Maxwell {widths}", spec=spec)


@pytest.mark.parametrize("pde,widths", [(PDE_BURGERS, [64, 64, 64]), (PDE_ALLEN_CAHN, [32, 224])])
def test_mma_output_kernel_one_output(cuda_lib, pde, widths):
    spec, p, B, b = _case(pde, 2, 1, widths, 0, 650, 90, 110, 321)
    prob = Problem(0.01, 1.0, 4.0, 2.0)
    gt, gg = run_gpu(spec, p, B, b, prob, "bf16")
    rt, rg = run_oracle(spec, p, B, b, prob)
    assert_parity(gt, gg, rt, rg, TOL["bf16"], f"one output {widths}", spec=spec)


@pytest.mark.parametrize("widths", [[64, 288], [32, 512]])
def test_tma_output_kernel_wider_layers(cuda_lib, widths):
    spec, p, B, b = _case(PDE_NS, 2, 3, widths, 16, 600, 0, 140, 331)
    gt, gg = run_gpu(spec, p, B, b, Problem(0.02, 1.0, 1.0, 1.0), "bf16")
    rt, rg = run_oracle(spec, p, B, b, Problem(0.02, 1.0, 1.0, 1.0))
    assert_parity(gt, gg, rt, rg, TOL["bf16"], f"NS {widths}", spec=spec)


@pytest.mark.parametrize("widths", [[64, 40], [48, 200]])
def test_register_output_kernel_other_widths(cuda_lib, widths):
    spec, p, B, b = _case(PDE_MAXWELL, 3, 3, widths, 0, 400, 60, 90, 341)
    gt, gg = run_gpu(spec, p, B, b, Problem(0.0, 1.0, 1.0, 1.0), "bf16")
    rt, rg = run_oracle(spec, p, B, b, Problem(0.0, 1.0, 1.0, 1.0))
    assert_parity(gt, gg, rt, rg, TOL["bf16"], f"Maxwell {widths}", spec=spec)


@pytest.mark.parametrize("pde,activation,n_res", [
    ("burgers", "tanh", 48500), ("burgers", "tanh", 48700),   # 760 blocks: the line between the two register limits
    ("ns", "sine", 29100), ("ns", "sine", 29200),             # 456 blocks
    ("ns", "tanh", 38800), ("ns", "tanh", 39000),             # 608 blocks: two rounds either way from here on
    ("ns", "tanh", 200), ("burgers", "sine", 200),
])
def test_output_kernel_register_limits(cuda_lib, pde, activation, n_res):
    """The CUDA-core output kernel on both sides of the rule that chooses its register limit."""
    code, d_out = (PDE_BURGERS, 1) if pde == "burgers" else (PDE_NS, 3)
    spec = NetSpec(code, 2, d_out, [12, 20], rwf=True)
    spec.activation, spec.omega0 = activation, 1.5
    p, prob = init_params(spec, 61, 0.2), Problem(0.02, 0.3, 2.0, 5.0)
    b = make_batch(code, n_res, 10 if d_out == 1 else 0, 20, 62, 63)
    gt, gg = run_gpu(spec, p, None, b, prob, "fp32")
    rt, rg = run_oracle(spec, p, None, b, prob, chunk=16384)
    assert_parity(gt, gg, rt, rg, TOL["fp32"], f"{pde} {activation} {n_res}", spec=spec)


@pytest.mark.parametrize("width,precision", [(13, "fp32"), (64, "bf16"), (288, "bf16"), (600, "bf16")])
def test_one_causal_segment_without_decay_is_the_plain_loss(cuda_lib, width, precision):
    """With one segment and eps = 0 the causal pass sums the plain loss (the plain kernels add up to
    four points in FP32 first: 3 roundings), and the gradient is the plain one bit for bit."""
    import torch
    from paper_2604_15645_gb300 import api
    spec = NetSpec(PDE_BURGERS, 2, 1, [16, width])
    params = torch.tensor(init_params(spec, 51, 0.2), device="cuda")
    db, prob = api.DeviceBatch.from_host(make_batch(PDE_BURGERS, 5000, 40, 30, 52, 53)), api.make_problem(0.05, 0.7, 0.5, 2.0)
    plain, causal = (api.PinnNet.from_spec(spec, precision) for _ in range(2))
    causal.set_causal(1, 0.0)
    t0, g0 = plain.loss_grad(params, db, prob)
    t1, g1 = causal.loss_grad(params, db, prob)
    torch.cuda.synchronize()
    assert plain.status_poll() == 0 and causal.status_poll() == 0
    assert torch.allclose(t0, t1, rtol=2.0 ** -22, atol=0.0)
    assert torch.equal(g0, g1)
