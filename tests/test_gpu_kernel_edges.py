"""Kernels at the sizes where their tiling can go wrong (tile edges, remainders, the
smallest and largest of a dispatch rule's range), against the FP64 oracle at the
precision's stated tolerance."""
import numpy as np
import pytest
import torch

from synth import NetSpec, Problem, ff_matrix, init_params, make_batch
from synth.workloads import PDE_BURGERS, PDE_MAXWELL, PDE_NS

from gpu_helpers import TOL, assert_parity, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def _parity(spec, n_res, n_ic, n_bc, precision, what):
    p = init_params(spec, 71, 0.2)
    B = ff_matrix(spec, 72)
    b = make_batch(spec.pde, n_res, n_ic, n_bc, 73, 74)
    prob = Problem(0.02, 0.3, 2.0, 5.0)
    gt, gg = run_gpu(spec, p, B, b, prob, precision)
    rt, rg = run_oracle(spec, p, B, b, prob, chunk=4096)
    assert_parity(gt, gg, rt, rg, TOL[precision], what, spec=spec)


@pytest.mark.parametrize("widths,ff,n_res", [
    ([1, 3], 0, 1),                # a single point; 4-byte weight copies; one K step, mostly padding
    ([66, 130, 17], 5, 95),        # widths past a 64- and a 128-feature block, M not a multiple of 4
    ([64, 128, 64], 8, 4096),      # full blocks, 64-feature blocks at this size
    ([80, 72], 24, 9800),          # the smallest sizes that take 128-feature blocks
    ([64], 32, 30000),             # long weight-gradient splits (the narrow form of the kernel's sums)
])
def test_fp32_gemm_edges(cuda_lib, widths, ff, n_res):
    spec = NetSpec(PDE_NS, 2, 3, widths, ff_m=ff, ff_sigma=1.0, rwf=True)
    _parity(spec, n_res, 0, 33, "fp32", f"fp32 {widths} {n_res}")


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("pde,widths,n", [
    (PDE_BURGERS, [40, 16], (61, 2, 1)),          # one feature per thread, sets meeting inside a 4- or 8-point group
    (PDE_MAXWELL, [104, 16], (20003, 501, 77)),   # several features per thread, a remainder of them
])
def test_first_layer_edges(cuda_lib, pde, widths, n, precision):
    spec = NetSpec(pde, 3 if pde == PDE_MAXWELL else 2, 3 if pde == PDE_MAXWELL else 1, widths, rwf=True)
    _parity(spec, *n, precision, f"first layer {widths} {n} {precision}")


@pytest.mark.parametrize("precision,width", [("fp32", 13), ("bf16", 64), ("bf16", 320)])
@pytest.mark.parametrize("segments,n_res", [(32, 1000), (5, 3)])
def test_causal_segment_sums(cuda_lib, precision, width, segments, n_res):
    """All 32 segments, and segments without points, in each of the three output kernels."""
    import oracle
    from paper_2604_15645_gb300 import api
    spec = NetSpec(PDE_BURGERS, 2, 1, [width, width])
    p = init_params(spec, 81, 0.2)
    b = make_batch(PDE_BURGERS, n_res, 40, 30, 82, 83)
    net = api.PinnNet.from_spec(spec, precision)
    net.set_causal(segments, 1.5)
    t, g = net.loss_grad(torch.tensor(p, device="cuda"), api.DeviceBatch.from_host(b), api.make_problem(0.05, 1.0, 0.5, 2.0))
    torch.cuda.synchronize()
    assert net.status_poll() == 0
    cz = dict(segments=segments, eps=1.5, t_index=1, t0=0.0, t1=1.0)
    terms, rg = oracle.loss_and_grad(oracle.Model.from_spec(spec), p, None, b, 0.05, (1.0, 0.5, 2.0), causal=cz)
    tol = TOL[precision]
    t = t.cpu().numpy()
    assert abs(t[0] - terms["total"]) <= tol * abs(terms["total"])
    assert abs(t[1] - terms["pde"]) <= tol * abs(terms["pde"])
    assert np.linalg.norm(g.cpu().numpy() - rg) <= tol * np.linalg.norm(rg)
    assert np.allclose(net.causal_weights().cpu().numpy(), terms["causal_weights"], rtol=10 * tol)


@pytest.mark.parametrize("widths,ff", [
    ([16, 16], 0),                    # one GEMM layer, a quarter of a K chunk
    ([128, 72, 128], 64),             # at most 128 wide: two column tiles in flight
    ([136, 24, 256, 16, 200], 8),     # m-tiles of 136 and 200 rows, layers with one m-tile in between
    ([256, 256], 128),                # full 256
])
@pytest.mark.parametrize("n_res", [1, 20000])   # one tile, and more tiles than two rounds of every SM
def test_fused_forward_edges(cuda_lib, widths, ff, n_res):
    """The one-kernel forward gives bitwise the losses and gradients of the per-layer
    launches (which the grouped many-network step runs; those are checked against the
    oracle elsewhere), and a loss-only call gives the same loss."""
    from paper_2604_15645_gb300 import api
    spec = NetSpec(PDE_BURGERS, 2, 1, widths, ff_m=ff, ff_sigma=1.0, rwf=True)
    p, B = init_params(spec, 91, 0.2), ff_matrix(spec, 92)
    b = make_batch(PDE_BURGERS, n_res, 30, 20, 93, 94)
    prob, db = api.make_problem(0.02), api.DeviceBatch.from_host(b)
    params = torch.tensor(p, device="cuda")
    Bd = None if B is None else torch.tensor(B, device="cuda")
    res = []
    for grouped in (False, True):
        multi = api.PinnMulti([spec], "bf16")
        if Bd is not None:
            api._lib.check_multi(api._lib.load().pinn_multi_set_ff_matrix(multi.h, 0, Bd.data_ptr()), multi.h)
        multi.set_inputs([db], [prob])
        multi.grouped = grouped
        q = params.clone()
        grad, m, v = (torch.zeros_like(q) for _ in range(3))
        loss = multi.train_step(q, grad, m, v, step=1)
        torch.cuda.synchronize()
        assert multi.status_poll() == 0
        res.append((loss[0].clone(), grad))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    net = api.PinnNet.from_spec(spec, "bf16")
    if Bd is not None:
        net.set_ff_matrix(B)
    assert torch.equal(net.loss(params, db, prob), res[0][0])


@pytest.mark.parametrize("pde,widths,ff", [
    (PDE_BURGERS, [264, 272], 0),             # m-tiles of 8 rows, raw first layer (coordinate terms)
    (PDE_NS, [512, 304, 264], 16),            # even and odd m-tile counts
    (PDE_MAXWELL, [40, 1024, 16], 0),         # one m-tile below a wide layer, K of 16 chunks
])
@pytest.mark.parametrize("n_res", [1, 7000])  # one tile, and more units than two rounds of every SM
@pytest.mark.parametrize("value_split", [False, True])
def test_wide_layer_edges(cuda_lib, pde, widths, ff, n_res, value_split):
    """The per-layer forward and the staged adjoint of layers above 256 wide against the oracle:
    total loss and whole gradient (the residual of a single point may cancel below the
    precision's tolerance)."""
    spec = NetSpec(pde, 3 if pde == PDE_MAXWELL else 2, 1 if pde == PDE_BURGERS else 3, widths, ff_m=ff, ff_sigma=1.0)
    p, B, prob = init_params(spec, 95, 0.2), ff_matrix(spec, 96), Problem(0.02, 0.3, 2.0, 5.0)
    b = make_batch(pde, n_res, 30, 20, 97, 98)
    gt, gg = run_gpu(spec, p, B, b, prob, "bf16", value_split=value_split)
    rt, rg = run_oracle(spec, p, B, b, prob, chunk=4096)
    assert abs(gt[0] - rt[0]) <= TOL["bf16"] * abs(rt[0])
    assert np.linalg.norm(gg - rg) <= TOL["bf16"] * np.linalg.norm(rg)


@pytest.mark.parametrize("widths,ff", [
    ([512, 256, 264], 0),             # layers of four and two m-tiles (in pairs), then three (not)
    ([200, 1024, 136], 24),           # two m-tiles with a ragged second one, eight, K tails
])
@pytest.mark.parametrize("n_res", [1, 7000])
def test_paired_forward_edges(cuda_lib, widths, ff, n_res):
    """The forward in pairs of CTAs gives bitwise the loss and gradient of the unpaired launches
    (which the grouped many-network step runs)."""
    from paper_2604_15645_gb300 import api
    spec = NetSpec(PDE_MAXWELL, 3, 3, widths, ff_m=ff, ff_sigma=1.0, rwf=True)
    p, B = init_params(spec, 91, 0.2), ff_matrix(spec, 92)
    db = api.DeviceBatch.from_host(make_batch(PDE_MAXWELL, n_res, 30, 20, 93, 94))
    Bd = None if B is None else torch.tensor(B, device="cuda")
    res = []
    for grouped in (False, True):
        multi = api.PinnMulti([spec], "bf16")
        if Bd is not None:
            api._lib.check_multi(api._lib.load().pinn_multi_set_ff_matrix(multi.h, 0, Bd.data_ptr()), multi.h)
        multi.set_inputs([db], [api.make_problem(0.02)])
        multi.grouped = grouped
        q = torch.tensor(p, device="cuda")
        grad, m, v = (torch.zeros_like(q) for _ in range(3))
        loss = multi.train_step(q, grad, m, v, step=1)
        torch.cuda.synchronize()
        assert multi.status_poll() == 0
        res.append((loss[0].clone(), grad))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])


@pytest.mark.parametrize("pde,widths,ff", [
    (PDE_NS, [136, 24, 200], 8),      # ragged m-tiles and K blocks
    (PDE_BURGERS, [72, 264], 0),      # raw first layer (coordinate terms), three m-tiles
])
@pytest.mark.parametrize("n_res", [1, 7000])
def test_tf32_edges(cuda_lib, pde, widths, ff, n_res):
    """The TF32 epilogues against the oracle.  Bound: the weight gradient truncates both operands
    to 10 mantissa bits, at most 2^-10 of each."""
    spec = NetSpec(pde, 2, 1 if pde == PDE_BURGERS else 3, widths, ff_m=ff, ff_sigma=1.0)
    p, B, prob = init_params(spec, 81, 0.2), ff_matrix(spec, 82), Problem(0.02, 0.3, 2.0, 5.0)
    b = make_batch(pde, n_res, 30, 20, 83, 84)
    gt, gg = run_gpu(spec, p, B, b, prob, "tf32")
    rt, rg = run_oracle(spec, p, B, b, prob, chunk=4096)
    assert abs(gt[0] - rt[0]) <= TOL["tf32"] * abs(rt[0])
    assert np.linalg.norm(gg - rg) <= 2.0 ** -9 * np.linalg.norm(rg)


@pytest.mark.parametrize("widths,precision", [([13, 13], "fp32"), ([64, 64], "bf16"), ([8, 288], "bf16")])
def test_causal_segment_sums_beyond_fp32(cuda_lib, widths, precision):
    """A segment whose squared residuals are FP32 numbers but whose sum is not, in each of the
    three output kernels: the loss stays finite, the later segment's weight is 0 and no NaN."""
    import oracle
    from paper_2604_15645_gb300 import api
    from parity_blocks import param_blocks
    spec = NetSpec(PDE_BURGERS, 2, 1, widths)
    p = init_params(spec, 81, 0.2)
    b = make_batch(PDE_BURGERS, 2000, 40, 30, 82, 83)
    cz = dict(segments=2, eps=1.5, t_index=1, t0=0.0, t1=1.0)
    last = slice(*{n: (s, e) for n, s, e in param_blocks(spec)}["V3"][:2])

    def ref(scale):
        q = np.array(p, dtype=np.float32)
        q[last] *= scale
        return q, *oracle.loss_and_grad(oracle.Model.from_spec(spec), q, None, b, 0.05, (0.01, 0.0, 0.0), causal=cz)

    # u u_x is all of the residual: scale the output layer to a mean square of 4e37 in the
    # first segment (the sums of its points among a warp's 16 reach 5e38 to 7e38, no point 1.2e38)
    _, t, _ = ref(1e9)
    q, terms, rg = ref(np.float32(1e9 * (2e37 / t["pde"]) ** 0.25))   # pde = half of that mean
    assert list(terms["causal_weights"]) == [1.0, 0.0]
    net = api.PinnNet.from_spec(spec, precision)
    net.set_causal(2, 1.5)
    out, g = net.loss_grad(torch.tensor(q, device="cuda"), api.DeviceBatch.from_host(b), api.make_problem(0.05, 0.01, 0.0, 0.0))
    torch.cuda.synchronize()
    assert net.status_poll() == 0
    tol = TOL[precision]
    assert abs(float(out[0]) - terms["total"]) <= tol * terms["total"]
    assert net.causal_weights().cpu().tolist() == [1.0, 0.0]
    assert np.linalg.norm(g.cpu().numpy().astype(np.float64) - rg) <= tol * np.linalg.norm(rg)


@pytest.mark.parametrize("widths,value_split", [
    ([512, 1000, 256], False),        # eight m-tiles, the last of 104 rows; two on a K of 15.6 chunks
    ([384, 512, 200], True),          # four m-tiles; two, the second of 72 rows
])
def test_paired_forward_sizes(cuda_lib, monkeypatch, widths, value_split):
    """The forward in pairs of CTAs, at sizes that its dispatch gives it, bitwise against the
    unpaired launches (which the grouped many-network step runs)."""
    from paper_2604_15645_gb300 import _lib, api
    spec = NetSpec(PDE_MAXWELL, 3, 3, widths, rwf=True)
    p, n_res = init_params(spec, 91, 0.2), 30100
    db = api.DeviceBatch.from_host(make_batch(PDE_MAXWELL, n_res, 30, 20, 93, 94))
    prob = api.make_problem(0.02)
    net = api.PinnNet.from_spec(spec, "bf16", value_split=value_split)
    loss, grad = net.loss_grad(torch.tensor(p, device="cuda"), db, prob)
    make_spec, flags = _lib.make_spec, _lib.PINN_FLAG_BF16_VALUE_SPLIT if value_split else 0
    monkeypatch.setattr(_lib, "make_spec", lambda *args: make_spec(*args, flags))
    multi = api.PinnMulti([spec], "bf16")
    multi.set_inputs([db], [prob])
    multi.grouped = True
    q = torch.tensor(p, device="cuda")
    g, m, v = (torch.zeros_like(q) for _ in range(3))
    ref = multi.train_step(q, g, m, v, step=1)
    torch.cuda.synchronize()
    assert net.status_poll() == 0 and multi.status_poll() == 0
    assert torch.equal(loss, ref[0]) and torch.equal(grad, g)


@pytest.mark.parametrize("widths,ff", [([136, 256], 0), ([200], 64), ([64, 16], 0)])
@pytest.mark.parametrize("n_res", [1, 20000])
def test_single_gemm_layer(cuda_lib, widths, ff, n_res):
    """One hidden GEMM layer runs its own forward launch: bitwise the grouped launch's loss and
    gradient, and the same loss without a gradient."""
    from paper_2604_15645_gb300 import api
    spec = NetSpec(PDE_BURGERS, 2, 1, widths, ff_m=ff, ff_sigma=1.0, rwf=True)
    p, B = init_params(spec, 91, 0.2), ff_matrix(spec, 92)
    prob, db = api.make_problem(0.02), api.DeviceBatch.from_host(make_batch(PDE_BURGERS, n_res, 30, 20, 93, 94))
    Bd = None if B is None else torch.tensor(B, device="cuda")
    multi = api.PinnMulti([spec], "bf16")
    net = api.PinnNet.from_spec(spec, "bf16")
    if Bd is not None:
        api._lib.check_multi(api._lib.load().pinn_multi_set_ff_matrix(multi.h, 0, Bd.data_ptr()), multi.h)
        net.set_ff_matrix(B)
    multi.set_inputs([db], [prob])
    multi.grouped = True
    q = torch.tensor(p, device="cuda")
    g, m, v = (torch.zeros_like(q) for _ in range(3))
    ref = multi.train_step(q, g, m, v, step=1)
    params = torch.tensor(p, device="cuda")
    terms, grad = net.loss_grad(params, db, prob)
    terms = terms.clone()
    loss = net.loss(params, db, prob)
    torch.cuda.synchronize()
    assert net.status_poll() == 0 and multi.status_poll() == 0
    assert torch.equal(terms, ref[0]) and torch.equal(grad, g) and torch.equal(loss, terms)


@pytest.mark.parametrize("pde", [PDE_BURGERS, PDE_NS, PDE_MAXWELL])
@pytest.mark.parametrize("width", [64, 320])   # every layer in one kernel; layer by layer
def test_packed_forward_rule_matches_the_scalar_one(cuda_lib, pde, width):
    """The tensor-core epilogues' packed tanh-jet rule against the scalar rule of the CUDA-core
    kernels, on layers whose products and sums are exact in both (one power of two per row): the
    same losses bit for bit."""
    from paper_2604_15645_gb300 import _lib, api
    from parity_blocks import param_blocks
    d_in, d_out = (3, 3) if pde == PDE_MAXWELL else (2, 1 if pde == PDE_BURGERS else 3)
    spec = NetSpec(pde, d_in, d_out, [width] * 3)
    p = init_params(spec, 31, 0.2).astype(np.float32)
    rng = np.random.default_rng(32)
    blocks = {n: (s, e) for n, s, e in param_blocks(spec)}
    for name in ("V2", "V3"):
        W = np.zeros((width, width), np.float32)
        W[np.arange(width), rng.permutation(width)] = 2.0 ** rng.integers(-2, 5, width) * rng.choice([-1, 1], width)
        p[slice(*blocks[name])] = W.ravel()
    db = api.DeviceBatch.from_host(make_batch(pde, 6000, 0 if pde == PDE_NS else 50, 60, 33, 34))
    prob, params = api.make_problem(0.02, 0.5, 1.0, 2.0), torch.tensor(p, device="cuda")
    res = []
    for flags in (0, _lib.PINN_FLAG_CUDA_CORES):
        net = api.PinnNet.from_spec(spec, "bf16")
        _lib.pinn_destroy(net.h)
        net.h = _lib.pinn_create(_lib.make_spec(pde, spec.widths, 0, False, _lib.PRECISIONS["bf16"], flags))
        res.append(net.loss(params, db, prob).clone())
        torch.cuda.synchronize()
        assert net.status_poll() == 0
    assert torch.equal(res[0], res[1])


@pytest.mark.parametrize("n_res", [38879, 38880])
def test_fp32_weight_gradient_forms(cuda_lib, n_res):
    """One 64 x 64 weight-gradient tile in 608 splits: 256 columns each (the last size of the
    four-column form) and 288 (the first of the eight-column one), on 152 SMs."""
    spec = NetSpec(PDE_NS, 2, 3, [64], ff_m=32, ff_sigma=1.0, rwf=True)
    _parity(spec, n_res, 0, 33, "fp32", f"fp32 weight gradient, {n_res} points")


@pytest.mark.parametrize("pde,widths,ff", [(PDE_NS, [136, 24, 200], 8), (PDE_BURGERS, [72, 264], 0)])
@pytest.mark.parametrize("n_res", [1, 7000])
def test_tf32_edges_per_block(cuda_lib, pde, widths, ff, n_res):
    """The TF32 epilogues at the precision's stated tolerance, per loss term and per block of the
    gradient."""
    spec = NetSpec(pde, 2, 1 if pde == PDE_BURGERS else 3, widths, ff_m=ff, ff_sigma=1.0)
    p, B, prob = init_params(spec, 81, 0.2), ff_matrix(spec, 82), Problem(0.02, 0.3, 2.0, 5.0)
    b = make_batch(pde, n_res, 30, 20, 83, 84)
    gt, gg = run_gpu(spec, p, B, b, prob, "tf32")
    rt, rg = run_oracle(spec, p, B, b, prob, chunk=4096)
    assert_parity(gt, gg, rt, rg, TOL["tf32"], f"tf32 {widths} {n_res}", spec=spec)


@pytest.mark.parametrize("pde,widths,ff", [
    (PDE_BURGERS, [264, 272], 0), (PDE_NS, [512, 304, 264], 16), (PDE_MAXWELL, [40, 1024, 16], 0)])
def test_wide_layer_edges_per_block(cuda_lib, pde, widths, ff):
    """Layers above 256 wide, full split of the weights: per loss term and per block of the gradient."""
    spec = NetSpec(pde, 3 if pde == PDE_MAXWELL else 2, 1 if pde == PDE_BURGERS else 3, widths, ff_m=ff, ff_sigma=1.0)
    p, B, prob = init_params(spec, 95, 0.2), ff_matrix(spec, 96), Problem(0.02, 0.3, 2.0, 5.0)
    b = make_batch(pde, 7000, 30, 20, 97, 98)
    gt, gg = run_gpu(spec, p, B, b, prob, "bf16")
    rt, rg = run_oracle(spec, p, B, b, prob, chunk=4096)
    assert_parity(gt, gg, rt, rg, TOL["bf16"], f"bf16 {widths}", spec=spec)
