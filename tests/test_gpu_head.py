"""The head unit's write-back at each way a lane's codes lie in a row (parts of words; one or two whole bytes
for 4 and 8 bits), each state shape, and intervals of one, several and an uneven number of tokens, whose
inputs are loaded a token ahead, in lockstep with the oracle and under its bounds.  Unpack of every width bit
for bit, to dense states at every alignment; its layout check."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402
from test_gpu_parity import _lockstep  # noqa: E402

SHAPES = [(128, 128), (128, 64), (64, 64)]


@pytest.mark.parametrize("dk,dv", SHAPES)
@pytest.mark.parametrize("width", [1, 3, 4, 5, 7, 8, 9, 15, 16])
def test_head_widths(qs, orc, dk, dv, width):
    w = synth.scaled(synth.WORKLOADS["gdn_decode"], B=2, H=2, T=3, dk=dk, dv=dv, bbar=width,
                     bmin=width, bmax=width)
    _lockstep(qs, orc, w)


@pytest.mark.parametrize("dk,dv", SHAPES)
@pytest.mark.parametrize("name", ["gdn_decode", "gdn_general"])
@pytest.mark.parametrize("T,C,log_decay", [(7, 2, False), (11, 16, True), (21, 5, False)])
def test_head_intervals(qs, orc, dk, dv, name, T, C, log_decay):
    w = synth.scaled({**synth.WORKLOADS, **synth.EXTENSION_WORKLOADS}[name], B=2, H=3, T=T, C=C, dk=dk, dv=dv,
                     gate_bits=2 if log_decay else 0)
    _lockstep(qs, orc, w, log_decay=log_decay)


@pytest.mark.parametrize("dk,dv", SHAPES)
@pytest.mark.parametrize("pad", [0, 1, 2, 4])
def test_head_unpack(qs, orc, dk, dv, pad):
    H, total = 17, 17 * 8   # heads of widths 0 to 16
    kw = dict(B=2, H=H, dk=dk, dv=dv, decay_kind=1, unit_kind=1, bmin=0, bmax=16)
    cq, co = qs.Config(bbar_num=8, bbar_den=1, **kw), orc.Cfg(bbar_num=8, **kw)
    rng = np.random.default_rng(dk + dv + pad)
    w = np.stack([rng.permutation(17) for _ in range(2)])
    assert (w.sum(1) == total).all()
    nb = w * (dk * dv // 8)
    off = np.concatenate([np.zeros((2, 1), int), np.cumsum(nb, 1)[:, :-1]], 1)
    widths, off = w.astype(np.uint8).ravel(), off.astype(np.uint32).ravel()
    st = qs.new_state(cq)
    payload = rng.integers(0, 256, st.payload.numel(), dtype=np.uint8)
    scales = rng.lognormal(0, 2, st.scales.numel()).astype(np.float16).view(np.uint16)
    st.payload.copy_(torch.from_numpy(payload).view(st.payload.shape))
    st.scales.copy_(torch.from_numpy(scales.view(np.int16)).view(st.scales.shape).view(st.scales.dtype))
    st.widths.copy_(torch.from_numpy(widths))
    st.head_off.copy_(torch.from_numpy(off.view(np.int32)))
    n = 2 * H * dk * dv
    buf = torch.full((n + pad + 4,), 7.0, device="cuda")
    out = buf[pad:pad + n].view(2, H, dk, dv)
    qs.qstate_unpack(cq, st, out)
    qs.qstate_check()
    assert np.array_equal(out.cpu().numpy(), orc.unpack(co, payload, scales, widths, off))
    assert bool((buf[:pad] == 7).all()) and bool((buf[pad + n:] == 7).all())
    # a head whose rows would end past the region: reported, and the check is clean again afterwards
    st.head_off[H - 1] = st.payload.numel() // 2 - 16
    st.widths[H - 1] = 16
    qs.qstate_unpack(cq, st, out)
    with pytest.raises(qs.QstateError):
        qs.qstate_check()
    qs.qstate_check()
