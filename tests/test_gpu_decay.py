"""The decay-gate quantiser at the edges of its walks: channel counts that are multiples of 128, of 64
only, that divide 128, others up to 256 and above; 2 to 256 levels; few and odd numbers of rows; unaligned rates;
a rate that is not positive.  Codes bit for bit against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("row,H,dk", [(1, 1, 64), (1, 3, 64), (1, 2, 128), (1, 5, 128), (0, 1, 128), (0, 4, 128),
                                      (0, 2, 64), (0, 7, 128), (0, 12, 128), (0, 16, 128), (0, 61, 64), (0, 64, 64),
                                      (0, 192, 64), (0, 250, 64), (0, 256, 64), (0, 257, 64)])
@pytest.mark.parametrize("g", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("B,T,pad", [(1, 1, 0), (2, 37, 0), (1, 641, 0), (3, 5, 1)])
def test_quant_decay_walks(qs, orc, row, H, dk, g, B, T, pad):
    cfg = qs.Config(B=B, H=H, dk=dk, dv=64, decay_kind=0 if row else 1, unit_kind=0 if row else 1, gate_bits=g)
    shape = (B, T, H, dk) if row else (B, T, H)
    chan, L = (H * dk if row else H), 1 << g
    rng = np.random.default_rng(H * 100 + g + T)
    s = np.logaddexp(0, rng.normal(-2, 1, shape)).astype(np.float32)
    buf = torch.zeros(s.size + pad, device="cuda")
    buf[pad:] = torch.from_numpy(s.reshape(-1)).cuda()
    sd = buf[pad:].view(shape)
    code = torch.full((s.size + 8,), 77, dtype=torch.uint8, device="cuda")
    lut, thr = torch.zeros(chan * L, device="cuda"), torch.zeros(chan * (L - 1), device="cuda")
    qs.qstate_quant_decay(cfg, sd, code, lut, thr)
    qs.qstate_check()
    cref, lref, tref = orc.quant_decay(s, chan, g)
    assert np.array_equal(code[:s.size].cpu().numpy(), np.asarray(cref).reshape(-1))
    assert bool((code[s.size:] == 77).all())
    # levels and thresholds: FP64 on both sides, rounded to FP32 (their libraries' last bit)
    assert np.allclose(lut.cpu().numpy(), np.asarray(lref).reshape(-1), rtol=2.4e-7, atol=0)
    assert np.allclose(thr.cpu().numpy(), np.asarray(tref).reshape(-1), rtol=2.4e-7, atol=0)


@pytest.mark.parametrize("row,H", [(1, 3), (0, 16), (0, 12), (0, 7), (0, 257)])
@pytest.mark.parametrize("at", [-1, -3])
@pytest.mark.parametrize("bad", [0.0, -1.0, float("inf"), float("nan")])
def test_quant_decay_rejects_bad_rates(qs, row, H, at, bad):
    cfg = qs.Config(B=2, H=H, dk=128, dv=64, decay_kind=0 if row else 1, unit_kind=0 if row else 1, gate_bits=2)
    s = torch.rand((2, 9, H) + ((128,) if row else ()), device="cuda") + 0.1
    s.view(-1)[at] = bad
    chan = s[0, 0].numel()
    qs.qstate_quant_decay(cfg, s, torch.zeros(s.shape, dtype=torch.uint8, device="cuda"),
                          torch.zeros(chan * 4, device="cuda"), torch.zeros(chan * 3, device="cuda"))
    with pytest.raises(qs.QstateError):
        qs.qstate_check()
    qs.qstate_check()


@pytest.mark.parametrize("H", [260, 300, 516, 1000, 1020])
@pytest.mark.parametrize("g", [1, 2, 4, 5])
@pytest.mark.parametrize("B,T,pad", [(1, 1, 0), (1, 1023, 0), (2, 512, 0), (1, 1283, 0), (1, 1024, 1)])
def test_quant_decay_many_heads(qs, orc, H, g, B, T, pad):
    """Above 256 heads, in fours and from 1024 samples on: blocks in multiples of H / gcd(H, 1024), up to 255;
    others a rate at a time."""
    test_quant_decay_walks(qs, orc, 0, H, 64, g, B, T, pad)


@pytest.mark.parametrize("H", [260, 1020])
@pytest.mark.parametrize("at", [0, -1, 4567])
def test_quant_decay_many_heads_bad_rate(qs, H, at):
    cfg = qs.Config(B=1, H=H, dk=128, dv=64, decay_kind=1, unit_kind=1, gate_bits=2)
    s = torch.rand((1, 1040, H), device="cuda") + 0.1
    s.view(-1)[at] = -1.0
    qs.qstate_quant_decay(cfg, s, torch.zeros(s.shape, dtype=torch.uint8, device="cuda"),
                          torch.zeros(H * 4, device="cuda"), torch.zeros(H * 3, device="cuda"))
    with pytest.raises(qs.QstateError):
        qs.qstate_check()
    qs.qstate_check()
