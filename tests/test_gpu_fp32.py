"""qstate_scan_fp32 at the edges of its kernel: blocks of 8 staged tokens, 64-column CTAs, every
state shape, erasure and rate kind, unaligned inputs, against the FP64 recurrence (an FP32 readout of
128 terms, tokens' errors decaying with the state: 1e-5 relative, the bar of the FP32 tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def recur64(x, S, t0, t1):
    o = []
    for t in range(t0, t1):
        S = S * torch.exp(-x["s"][:, t].double()).reshape(S.shape[:2] + (-1, 1))
        k, v = x["k"][:, t].double(), x["v"][:, t].double()
        u = v
        if "a" in x:
            u = x["w"][:, t].double() * v - torch.einsum("bhi,bhij->bhj", x["a"][:, t].double(), S)
        elif "beta" in x:
            u = x["beta"][:, t].double()[..., None] * (v - torch.einsum("bhi,bhij->bhj", k, S))
        S = S + k[..., None] * u[..., None, :]
        o.append(torch.einsum("bhi,bhij->bhj", x["q"][:, t].double(), S))
    return torch.stack(o, 1), S


@pytest.mark.parametrize("dk,dv", [(128, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("erase", [0, 1, 2])
@pytest.mark.parametrize("rates", ["row", "head", "row_code", "head_code"])
@pytest.mark.parametrize("t0,t1,pad", [(0, 1, 0), (0, 8, 0), (3, 20, 0), (0, 17, 1)])
def test_scan_fp32(qs, dk, dv, erase, rates, t0, t1, pad):
    B, H, T = 2, 3, 20
    g = torch.Generator(device="cuda")
    g.manual_seed(dk + dv + erase + t1)

    def put(t):   # `pad` floats (bytes) off an allocation's 16-byte boundary
        flat = torch.zeros(t.numel() + pad, dtype=t.dtype, device="cuda")
        flat[pad:] = t.reshape(-1)
        return flat[pad:].view(t.shape)

    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    row = rates.startswith("row")
    x = dict(q=rnd(B, T, H, dk) / dk ** 0.5, k=rnd(B, T, H, dk) / dk ** 0.5, v=rnd(B, T, H, dv),
             s=torch.nn.functional.softplus(rnd(*((B, T, H, dk) if row else (B, T, H))) - 2))
    if erase == 0:
        x["beta"] = torch.sigmoid(rnd(B, T, H))
    elif erase == 2:
        x["a"], x["w"] = 0.5 * x["k"] + 0.1 * rnd(B, T, H, dk) / dk ** 0.5, torch.sigmoid(rnd(B, T, H, dv))
    x = {n: put(t) for n, t in x.items()}
    cfg = qs.Config(B=B, H=H, dk=dk, dv=dv, decay_kind=0 if row else 1, erase_kind=erase, C=4,
                    gate_bits=2 if "code" in rates else 0)
    X = qs.Inputs(x["q"], x["k"], x["v"], x["s"], None, None, x.get("beta"), T, x.get("a"), x.get("w"))
    if "code" in rates:
        chan = H * dk if row else H
        X.s_code = put(torch.zeros(x["s"].shape, dtype=torch.uint8, device="cuda"))
        X.s_lut = torch.zeros(chan * 4, device="cuda")
        qs.qstate_quant_decay(cfg, x["s"].contiguous(), X.s_code, X.s_lut, torch.zeros(chan * 3, device="cuda"))
        at = torch.arange(chan, device="cuda").view(x["s"].shape[2:]) * 4 + X.s_code.long()
        x["s"] = X.s_lut[at]
        X.s = None
    S0 = rnd(B, H, dk, dv)
    S = put(S0)
    o = put(torch.full((B, T, H, dv), 7.0, device="cuda"))
    qs.qstate_scan_fp32(cfg, S, X, t0, t1, o)
    qs.qstate_check()
    ref, Sref = recur64(x, S0.double(), t0, t1)
    rel = lambda y, z: float((y.double() - z).norm() / z.norm())  # noqa: E731
    assert rel(o[:, t0:t1], ref) < 1e-5 and rel(S, Sref) < 1e-5
    outside = torch.cat([o[:, :t0], o[:, t1:]], 1)
    assert bool((outside == 7.0).all())
    before = S.clone()
    qs.qstate_scan_fp32(cfg, S, X, t1, t1, o)   # no tokens
    assert torch.equal(S, before)


@pytest.mark.parametrize("dk,dv", [(128, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("erase", [0, 1, 2])
@pytest.mark.parametrize("rates", ["row", "head_code"])
@pytest.mark.parametrize("t0,t1,pad", [(0, 2, 0), (7, 8, 0), (7, 9, 0), (0, 3, 0), (0, 1, 1), (0, 2, 2)])
def test_few_tokens(qs, dk, dv, erase, rates, t0, t1, pad):
    """Calls of one or two tokens on an aligned state have a kernel of their own: both sides of that line."""
    test_scan_fp32(qs, dk, dv, erase, rates, t0, t1, pad)
