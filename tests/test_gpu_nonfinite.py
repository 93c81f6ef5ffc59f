"""Values that are not finite, or overflow, in one head's inputs: the write-back and the allocation after it
end, other heads of the write-back and other batch elements are bit for bit as without them."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402


@pytest.mark.parametrize("name,size,over", [("kda_decode", dict(H=4, T=3, C=3, gate_bits=0), {}),
                                            ("mamba2_decode", dict(H=4, T=1, group_heads=2), {}),
                                            ("gdn_decode", dict(H=4, T=3, C=3), {}),
                                            ("gdn_decode", dict(H=4, T=1, dk=64, dv=64), {}),
                                            ("kda_prefill", dict(H=4, T=40, C=40), dict(interval_form=1))],
                         ids=lambda v: str(v))
@pytest.mark.parametrize("array,value", [("v", float("nan")), ("v", float("inf")), ("k", float("nan")), ("k", 1e25),
                                         ("q", float("-inf")), ("v", 3e38)])
def test_one_head(qs, name, size, over, array, value):
    w = synth.scaled(synth.WORKLOADS[name], B=2, **size)
    cfg = qs.Config.from_workload(w, **over)
    b, h = 0, 2
    out = []
    for bad in (False, True):
        x = synth.device_inputs(w)
        if bad:
            x[array][b, w.T // 2, h, 5] = value
        X = qs.Inputs(x["q"], x["k"], x["v"], x["s"], None, None, x.get("beta"), w.T)
        A, B, st = qs.new_state(cfg), qs.new_state(cfg), qs.new_stats(cfg)
        o = torch.zeros((w.B, w.T, w.H, w.dv), device="cuda")
        S = torch.randn((w.B, w.H, w.dk, w.dv), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
        qs.qstate_init(cfg, A, B)
        qs.qstate_pack(cfg, S, A)
        qs.qstate_step(cfg, A, B, X, 0, w.T, 0, o, st)
        qs.qstate_check()
        D = torch.empty_like(S)
        qs.qstate_unpack(cfg, B, D)
        qs.qstate_check()
        budget = A.widths.view(w.B, -1).int().sum(1)   # the next allocation
        assert bool((budget == w.bbar * cfg.units).all())
        units = [t.view(w.B, w.H, -1) for t in (B.scales, B.fidx, st.ema_s, st.ema_r) + (() if w.unit == "head" else (st.range,))]
        out.append([o.transpose(1, 2), D] + units + [A.widths[cfg.units:], A.head_off[w.H:]])
    same = torch.ones((w.B, w.H), dtype=torch.bool, device="cuda")
    same[b, h] = False
    for good, bad in zip(*out):
        if good.dim() == 1:   # element 1's next widths and offsets
            assert torch.equal(good, bad)
        else:
            assert torch.equal(good[same], bad[same])
