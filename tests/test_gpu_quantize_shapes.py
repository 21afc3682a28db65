"""The quantisers' row-per-lanes kernels at every width class, ragged row counts and unaligned buffers, bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(1, 4), (33, 12), (100, 32), (17, 36), (1001, 64), (7, 68), (65, 128), (9, 132),
                                 (301, 256), (5, 260), (130, 512), (3, 516), (50, 1024)])
@pytest.mark.parametrize("shift", [0, 1])
def test_widths_and_alignment(n, d, shift):
    import torch

    import paper_2408_08933_gb300 as pkg

    rng = np.random.default_rng(n + d)
    X = rng.standard_normal((n, d)).astype(np.float32) * np.exp(rng.uniform(-20, 20, (n, 1))).astype(np.float32)
    X[n // 2] = 0.0
    buf = torch.empty(n * d + 1, dtype=torch.float32, device="cuda:0")
    Xd = buf[shift:shift + n * d].view(n, d)     # shift 1: four bytes off every wider boundary
    Xd.copy_(torch.from_numpy(X))
    got16, _ = pkg.quantize(Xd, "bf16")
    got8, gs = pkg.quantize(Xd, "fp8")
    torch.cuda.synchronize()
    ref8, rs = oracle.quant_e4m3(X)
    assert np.array_equal(got16.cpu().numpy().view(np.uint16), oracle.quant_bf16(X))
    assert np.array_equal(gs.cpu().numpy(), rs)
    assert np.array_equal(got8.cpu().numpy(), ref8)


@pytest.mark.parametrize("n,d", [(1, 4), (127, 4), (128, 4), (129, 4), (511, 4), (512, 4), (513, 4), (1003, 380), (64, 640)])
def test_bf16_block_edges(n, d):
    # blocks of 512 chunks of 4 elements: one short, full, one over, many
    import torch

    import paper_2408_08933_gb300 as pkg

    X = np.random.default_rng(n + d).standard_normal((n, d)).astype(np.float32)
    got, _ = pkg.quantize(torch.from_numpy(X).to("cuda:0"), "bf16")
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy().view(np.uint16), oracle.quant_bf16(X))
