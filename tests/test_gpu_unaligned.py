"""Write-backs whose arrays do not begin on a 16-byte boundary (views into larger tensors), in lockstep
with the oracle: such calls take the kernels without 16-byte copies and compute the same."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402
from test_gpu_parity import _lockstep  # noqa: E402

WORKLOADS = {**synth.WORKLOADS, **synth.EXTENSION_WORKLOADS}


class Shifted:
    """The binding with the named arrays one element past a 16-byte boundary."""

    def __init__(self, qs, *names):
        self.qs, self.names = qs, set(names)

    def __getattr__(self, name):
        return getattr(self.qs, name)

    def shift(self, obj):
        for n in self.names & set(vars(obj)):
            t = getattr(obj, n)
            if t is not None:
                buf = torch.zeros(t.numel() + 1, dtype=t.dtype, device=t.device)
                buf[1:] = t.reshape(-1)
                setattr(obj, n, buf[1:].view(t.shape))
                assert getattr(obj, n).data_ptr() % 16 == t.element_size()
        return obj

    def Inputs(self, *args):
        return self.shift(self.qs.Inputs(*args))

    def new_state(self, cfg):
        return self.shift(self.qs.new_state(cfg))

    def new_stats(self, cfg):
        return self.shift(self.qs.new_stats(cfg))


@pytest.mark.parametrize("dk,dv", [(128, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("name,array,C", [("kda_general", "a", 1), ("kda_general", "w", 3), ("kda_decode", "s_lut", 1),
                                          ("kda_decode", "s_lut", 5)])
def test_one_token_input(qs, orc, dk, dv, name, array, C):
    """a, w and the level table, which the 16-byte kernel copies too."""
    w = synth.scaled(WORKLOADS[name], B=2, H=3, T=10, C=C, dk=dk, dv=dv)
    _lockstep(Shifted(qs, array), orc, w, log_decay=array == "s_lut")


def test_level_table_chunked(qs, orc):
    """The chunked form copies the level table too: without its alignment the token form runs."""
    w = synth.scaled(WORKLOADS["kda_prefill"], B=1, H=2, T=70, C=48, gate_bits=2)
    _lockstep(Shifted(qs, "s_lut"), orc, w, log_decay=True, interval_form=1)


@pytest.mark.parametrize("dk,dv", [(128, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("head", [0, 1])
@pytest.mark.parametrize("pad", [1, 2, 3])
def test_dense_state(qs, dk, dv, head, pad):
    """Pack from and unpack to a dense state at any 4-byte alignment: as with an aligned one."""
    B, H = 2, 17
    cfg = qs.Config(B=B, H=H, dk=dk, dv=dv, decay_kind=head, unit_kind=head, bbar_num=8, bbar_den=1, bmin=0, bmax=16)
    gen = torch.Generator(device="cuda").manual_seed(dk + dv + pad)
    S = torch.randn((B, H, dk, dv), device="cuda", generator=gen)
    # widths 0 to 16, over the rows of a head or over the heads
    w = (torch.arange(17, dtype=torch.uint8).repeat(B) if head else
         torch.stack([torch.arange(dk) % 17 for _ in range(B * H)]).clamp(max=16).to(torch.uint8).reshape(-1))
    per_head = (w.view(B, H, -1).int().sum(2) * (dk * dv if head else dv) // 8).cpu()
    assert int(per_head.sum(1).max()) <= qs.region_bytes(cfg)
    off = torch.cumsum(per_head, 1).int() - per_head.int()
    got = []
    for p in (0, pad):
        st = qs.new_state(cfg)
        st.widths.copy_(w)
        st.head_off.copy_(off.reshape(-1))
        buf = torch.full((S.numel() + p + 4,), 7.0, device="cuda")
        view = buf[p:p + S.numel()].view(S.shape)
        view.copy_(S)
        qs.qstate_pack(cfg, view, st)
        view.fill_(0)
        qs.qstate_unpack(cfg, st, view)
        qs.qstate_check()
        assert bool((buf[:p] == 7).all()) and bool((buf[p + S.numel():] == 7).all())
        got.append((st.payload, st.scales, st.fidx, view.clone()))
    for a, b in zip(*got):
        assert torch.equal(a, b)


ARRAYS = {"token inputs": ("q", "k", "v", "s", "s_code", "beta", "a", "w"), "metadata": ("scales", "widths", "fidx"),
          "statistics": ("ema_s", "ema_r", "range")}


@pytest.mark.parametrize("dk,dv", [(128, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("name,gate_bits", [("kda_decode", 0), ("kda_decode", 2), ("kda_decode", 4), ("mamba2_decode", 0),
                                            ("kda_general", 0), ("gdn_decode", 0), ("gdn_decode", 3), ("gdn_general", 0)])
@pytest.mark.parametrize("arrays,C,fit_every", [("token inputs", 1, 1), ("metadata", 3, 1), ("statistics", 4, 3)])
def test_write_back(qs, orc, dk, dv, name, gate_bits, arrays, C, fit_every):
    """Everything but the payload off its boundary, row unit and head unit."""
    w = synth.scaled(WORKLOADS[name], B=2, H=4, T=9, C=C, dk=dk, dv=dv, group_heads=2 if "mamba" in name else 1,
                     gate_bits=gate_bits)
    _lockstep(Shifted(qs, *ARRAYS[arrays]), orc, w, log_decay=gate_bits > 0, fit_every=fit_every)
