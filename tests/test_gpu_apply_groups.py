"""hh_apply_multi on small lattices: one sweep over several vectors.

The groups' sweeps run the arithmetic of the single applies on the same
operands, so every vector must equal its own hh_apply bit for bit: at the
edges of a group (FP32 Q: 8 vectors, FP64 Q: 4), for each operator, group
width of x (N_x divisible by 4, 2, neither), and where vectors are not 16
bytes aligned (the per-vector path)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads  # noqa: E402


@pytest.fixture(scope="module")
def hh():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1007_3432_gb300 as pkg
    from paper_1007_3432_gb300 import build
    build.build()
    pkg.load()
    return pkg


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("op", ["M", "MT", "MTM"])
@pytest.mark.parametrize("d,nx,ntau", [(1, 32, 6), (1, 18, 4), (1, 7, 5), (1, 6, 3), (3, 4, 5), (3, 5, 4), (3, 6, 2)])
@pytest.mark.parametrize("k", [2, 4, 5, 8, 9])
def test_group_sweep_equals_single_applies(hh, d, nx, ntau, dtype, op, k):
    n = nx ** d * ntau
    code = {"M": hh.HH_OP_M, "MT": hh.HH_OP_MT, "MTM": hh.HH_OP_MTM}[op]
    x = torch.from_numpy(np.stack([workloads.source(n, seed=71, rhs=a) for a in range(k)])).to(dtype).cuda()
    with hh.Context(d, nx, ntau) as ctx:
        ctx.set_field(torch.from_numpy(workloads.sigma_field(n, seed=72)).cuda())
        y = torch.full_like(x, float("nan"))
        ctx.apply_multi(code, x, y, k)
        for v in range(k):
            xv, yv = x[v].clone(), torch.empty_like(x[v])
            ctx.apply(code, xv, yv)
            if d == 3 and nx % 4 == 0 and op == "MTM" and dtype == torch.float32:
                # the multi-vector kernel: another order of the sums
                assert torch.allclose(y[v], yv, rtol=1e-5, atol=1e-5)
            else:
                assert torch.equal(y[v], yv), v


@pytest.mark.parametrize("dtype,d,nx,ntau,k", [(torch.float64, 1, 1000, 900, 4), (torch.float64, 3, 21, 96, 4),
                                               (torch.float32, 1, 2000, 900, 5), (torch.float32, 3, 22, 180, 3)])
def test_group_sized_by_the_l2(hh, dtype, d, nx, ntau, k):
    """Lattices on which half of the L2 (x, t and y of 64 MiB), not the CG
    scratch, sets the group: two or three vectors, and a remainder."""
    n = nx ** d * ntau
    esz = 4 if dtype == torch.float32 else 8
    group = (64 << 20) // (3 * n * esz)
    assert 2 <= group < k <= 4 * 8 // esz and k % group != 0
    x = torch.from_numpy(np.stack([workloads.source(n, seed=73, rhs=a) for a in range(k)])).to(dtype).cuda()
    with hh.Context(d, nx, ntau) as ctx:
        ctx.set_field(torch.from_numpy(workloads.sigma_field(n, seed=74)).cuda())
        y = torch.full_like(x, float("nan"))
        ctx.counters_reset()
        ctx.apply_multi(hh.HH_OP_MTM, x, y, k)
        assert ctx.counters()["kernel_launches"] == 2 * ((k + group - 1) // group)
        for v in range(k):
            xv, yv = x[v].clone(), torch.empty_like(x[v])
            ctx.apply(hh.HH_OP_MTM, xv, yv)
            assert torch.equal(y[v], yv), v
