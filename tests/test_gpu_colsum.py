"""Column sums (bias gradients, weight gradient of the one-output layer) where their split over rows and columns can go
wrong: fewer rows than row lanes, one row, widths that fill no 64-byte piece."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2511_20564_b200 as E  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("f32", 4), ("f32", 20), ("f32", 72), ("bf16", 8), ("bf16", 40), ("bf16", 256)])
@pytest.mark.parametrize("rows", [1, 63, 64, 513, 4097])
def test_bias_gradient_of_the_gate(dtype, d, rows):
    rng = np.random.default_rng(rows * 1000 + d)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    alloc = (rows + 127) // 128 * 128
    mk = lambda r: torch.from_numpy(rng.standard_normal((r, d)).astype(np.float32)).to(dt).cuda()
    F, dFused, gate = mk(alloc), mk(alloc), torch.sigmoid(mk(alloc).float()).to(dt)
    Wg = mk(d) * 0.1
    ws = E.gate_fusion_forward(F, rows, Wg)[2]
    dbg = E.gate_fusion_backward(dFused, F, rows, gate, Wg, ws)[2]
    f, g, df = (t[:rows].double().cpu().numpy() for t in (F, gate, dFused))
    dpre = df * f * g * (1 - g)
    mass = np.abs(dpre).sum(0)
    # every term is rounded to the storage type (bf16: 8 significant bits, at most 2^-8 of the value) after four fp32
    # roundings, then added by 512 row lanes and a tree of 19
    bound = mass * ((2.0 ** -8 if dtype == "bf16" else 0.0) + (rows / 512 + 28) * 2.0 ** -24)
    err = np.abs(dbg.double().cpu().numpy() - dpre.sum(0))
    assert (err <= bound + 1e-30).all(), (err / bound).max()
