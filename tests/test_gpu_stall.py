"""Failure detection in the kernels of a whole pass, without a GPU fault: pinn_debug_stall launches
a handle's tcgen05 kernels with an arrival that never comes, under a 1 ms bound on every wait.
Every kernel of the pass must end through its abort path, the host must read
PINN_ERR_TIMEOUT, and the context must stay usable: the same call without the stall gives
the bits it gave before."""
import pytest
import torch

from synth import NetSpec, ff_matrix, init_params, make_batch
from synth.workloads import PDE_BURGERS, PDE_MAXWELL, PDE_NS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pde,widths,ff,n_res,precision,activation", [
    (PDE_BURGERS, [64, 48, 64], 0, 3000, "bf16", "tanh"),       # the one-kernel forward, two tiles in flight; fused adjoint
    (PDE_NS, [256, 200], 64, 3000, "bf16", "tanh"),             # two m-tiles
    (PDE_MAXWELL, [512, 512, 512], 0, 30000, "bf16", "tanh"),   # pairs of CTAs, staged adjoint, 256-row weight gradient
    (PDE_NS, [128, 264], 16, 3000, "tf32", "tanh"),
    (PDE_BURGERS, [64, 64], 16, 3000, "bf16", "sine"),
])
@pytest.mark.parametrize("graph", [False, True])
def test_every_kernel_of_a_pass_ends_by_itself(cuda_lib, pde, widths, ff, n_res, precision, activation, graph):
    from paper_2604_15645_gb300 import _lib, api
    d_in, d_out = (3, 3) if pde == PDE_MAXWELL else (2, 1 if pde == PDE_BURGERS else 3)
    spec = NetSpec(pde, d_in, d_out, widths, ff_m=ff, ff_sigma=1.0, activation=activation, omega0=2.0)
    net = api.PinnNet.from_spec(spec, precision)
    net.set_graph(graph)
    if ff:
        net.set_ff_matrix(ff_matrix(spec, 12))
    params, prob = torch.tensor(init_params(spec, 11, 0.2), device="cuda"), api.make_problem(0.02)
    db = api.DeviceBatch.from_host(make_batch(pde, n_res, 0 if pde == PDE_NS else 30, 40, 13, 14))
    assert _lib.pinn_tensor_core_layers(net.h, *db.sizes) == len(widths) - (0 if ff else 1)
    grad = torch.empty_like(params)

    def call():
        t, g = net.loss_grad(params, db, prob, grad=grad)
        torch.cuda.synchronize()
        return t.clone(), g.clone()

    before = call()
    assert net.status_poll() == 0
    for _ in range(2):
        _lib.pinn_debug_stall(net.h, 1000)
        call()
        assert net.status_poll() == 6                  # PINN_ERR_TIMEOUT
        _lib.pinn_debug_stall(net.h, 0)
        after = call()
        assert net.status_poll() == 0
        assert torch.equal(before[0], after[0]) and torch.equal(before[1], after[1])
    for us in (-1, 2000001):
        with pytest.raises(_lib.PinnError) as e:
            _lib.pinn_debug_stall(net.h, us)
        assert e.value.status == 1
