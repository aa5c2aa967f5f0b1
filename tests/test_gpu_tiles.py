"""GPU tests at the sizes where a kernel's tiling or its dispatch changes: tile edges, remainders, ends of the range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

hs = pytest.importorskip("paper_2609_24197_b200")


def _rand(shape, seed, dtype=torch.float16, std=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randn(shape, generator=g, device="cuda") * std).to(dtype)


# rows that make the 2-SM kernel take tiles of 256, 224, 192, 160 and 128 rows, full and with a remainder, whole waves and tail
# waves; weight rows that end inside a tile of the pair
@pytest.mark.parametrize("M,n_out,K", [(256, 256, 64), (257, 300, 520), (289, 1000, 512), (430, 2048, 1024), (448, 2048, 1024),
                                       (449, 512, 2048), (549, 4096, 1024), (640, 19200, 256), (1153, 1111, 264)])
@pytest.mark.parametrize("kind", ["f32", "accumulate", "f16"])
def test_many_row_gemm_tile_widths(M, n_out, K, kind):
    x, w = _rand((M, K), 1), _rand((n_out, K), 2, std=0.05)
    ref = x.double() @ w.double().t()
    y = torch.zeros((M, n_out), dtype=torch.float16 if kind == "f16" else torch.float32, device="cuda")
    if kind == "accumulate":
        y = _rand((M, n_out), 3, torch.float32)
        ref = ref + y.double()
    ws = torch.empty(hs.hspec_gemm_workspace_bytes(M, n_out, K), dtype=torch.uint8, device="cuda")
    hs.hspec_op_gemm(x, w, y, accumulate=kind == "accumulate", workspace=ws)
    # products of 16-bit values are exact in fp32; K additions of terms of size |x||w| round to 2^-24 of the running sum each
    # (bounded by the sum of magnitudes), the fp16 store to 2^-11 of the value
    mag = x.double().abs() @ w.double().abs().t() + ref.abs()
    bound = K * 2.0 ** -24 * mag + (2.0 ** -11 * ref.abs() + 1e-7 if kind == "f16" else 0.0)
    worst = float(((y.double() - ref).abs() / bound).max())
    assert worst <= 1.0, worst
