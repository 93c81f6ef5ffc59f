"""Row-unit pack and unpack at the edges of their kernels: every state shape, widths 0 to 16, a dense
state 8 but not 16 bytes aligned, values on a grid (many near ties between factors), offsets in
another order than the heads', NaN and infinity, inconsistent layouts; against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from parity import compare_packed, from_gpu_state, set_gpu_state  # noqa: E402

SHAPES = [(128, 128), (128, 64), (64, 64)]


def setup(qs, orc, dk, dv, reverse=False, bbar=5, B=2, H=3, seed=0):
    kw = dict(B=B, H=H, dk=dk, dv=dv, bmin=0, bmax=16)
    cq, co = qs.Config(bbar_num=bbar, bbar_den=1, **kw), orc.Cfg(bbar_num=bbar, **kw)
    rng = np.random.default_rng(seed)
    # rows of every width, the mean at most bbar, heads in index order or the other way round
    w = np.minimum(rng.integers(0, 17, (B, H, dk)), 16)
    while w.sum(axis=(1, 2)).max() > bbar * H * dk:
        w = np.maximum(w - rng.integers(0, 2, w.shape), 0)
    w[:, :, :17] = np.arange(17)
    w[:, :, 17:34] = 0
    nbytes = w.sum(2) * dv // 8
    assert (nbytes.sum(1) <= cq.H * dk * dv * bbar // 8).all()
    order = np.arange(H)[::-1] if reverse else np.arange(H)
    off = np.zeros((B, H), np.uint32)
    for b in range(B):
        at = 0
        for h in order:
            off[b, h] = at
            at += nbytes[b, h]
    return cq, co, w.astype(np.uint8).ravel(), off.ravel(), rng


def put(a, pad):
    flat = torch.zeros(a.size + pad, device="cuda")
    flat[pad:] = torch.from_numpy(a.ravel()).cuda()
    return flat[pad:].view(a.shape)


@pytest.mark.parametrize("dk,dv", SHAPES)
@pytest.mark.parametrize("values", ["normal", "grid"])
@pytest.mark.parametrize("pad", [0, 2])
def test_pack_unpack(qs, orc, dk, dv, values, pad):
    cq, co, widths, off, rng = setup(qs, orc, dk, dv, seed=dk + dv)
    S = rng.standard_normal((2, 3, dk, dv)) * np.exp(rng.uniform(-2, 2, (2, 3, dk, 1)))
    if values == "grid":
        S = np.round(S * 4) / 4
    S = S.astype(np.float32)
    S[0, 0, 3] = 0
    S[0, 0, 4] *= 1e-7     # FP16-subnormal steps
    S[0, 1, 5] *= 1e6      # steps at FP16's largest
    payload, scales, fidx, ranges = orc.pack(co, S, widths, off)
    ref = orc.Buf(payload, scales, widths, off, fidx)
    st = qs.new_state(cq)
    st.widths.copy_(torch.from_numpy(widths))
    st.head_off.copy_(torch.from_numpy(off.view(np.int32)))
    r = torch.zeros(widths.size, device="cuda")
    qs.qstate_pack(cq, put(S, pad), st, r)
    qs.qstate_check()
    gpu = from_gpu_state(orc, st)
    compare_packed(orc, co, gpu, ref, X=S)
    assert np.array_equal(r.cpu().numpy(), ranges)
    for buf in (ref, gpu):
        set_gpu_state(st, buf)
        out = put(np.zeros(S.shape, np.float32), pad)
        qs.qstate_unpack(cq, st, out)
        qs.qstate_check()
        assert np.array_equal(out.cpu().numpy(), orc.unpack(co, buf.payload, buf.scales, buf.widths, buf.head_off))


@pytest.mark.parametrize("dk,dv", SHAPES)
def test_heads_in_another_order(qs, orc, dk, dv):
    """Offsets that put the last head first: the same steps and values as in index order."""
    got = []
    for reverse in (False, True):
        cq, co, widths, off, rng = setup(qs, orc, dk, dv, reverse, seed=7)
        S = rng.standard_normal((2, 3, dk, dv)).astype(np.float32)
        st, D = qs.new_state(cq), torch.empty(S.shape, device="cuda")
        st.widths.copy_(torch.from_numpy(widths))
        st.head_off.copy_(torch.from_numpy(off.view(np.int32)))
        qs.qstate_pack(cq, torch.from_numpy(S).cuda(), st)
        qs.qstate_unpack(cq, st, D)
        qs.qstate_check()
        got.append((st.scales.cpu(), st.fidx.cpu(), D.cpu()))
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("dk,dv", SHAPES)
def test_pack_with_nan_and_infinity(qs, orc, dk, dv):
    """An infinity is its row's range; a NaN does not enter it and takes the lowest code; other rows
    are as without them."""
    cq, co, widths, off, rng = setup(qs, orc, dk, dv, seed=5)
    S = rng.standard_normal((2, 3, dk, dv)).astype(np.float32)
    S[1, 2, 9, 8] = 20.0
    out = []
    for bad in (False, True):
        X = S.copy()
        if bad:
            X[1, 2, 9, 7], X[0, 1, 8, 40] = np.nan, -np.inf
        st, r = qs.new_state(cq), torch.zeros(widths.size, device="cuda")
        st.widths.copy_(torch.from_numpy(widths))
        st.head_off.copy_(torch.from_numpy(off.view(np.int32)))
        qs.qstate_pack(cq, torch.from_numpy(X).cuda(), st, r)
        qs.qstate_check()
        D = torch.empty(X.shape, device="cuda")
        qs.qstate_unpack(cq, st, D)
        out.append((r.cpu().numpy().reshape(2, 3, dk), D.cpu().numpy()))
    (r0, d0), (r1, d1) = out
    assert np.isinf(r1[0, 1, 8]) and r1[1, 2, 9] == 20.0
    assert d1[1, 2, 9, 7] == d1[1, 2, 9].min() < -19
    same = np.ones((2, 3, dk), bool)
    same[1, 2, 9] = same[0, 1, 8] = False
    assert np.array_equal(r0[same], r1[same]) and np.array_equal(d0[same], d1[same])


@pytest.mark.parametrize("dk,dv", SHAPES)
@pytest.mark.parametrize("fault", ["width", "offset", "alignment"])
def test_inconsistent_layout_is_reported(qs, orc, dk, dv, fault):
    cq, co, widths, off, rng = setup(qs, orc, dk, dv, seed=6)
    widths, off = widths.copy(), off.copy()
    if fault == "width":
        widths[3] = 17
    else:
        off[4] += 4 if fault == "alignment" else cq.H * dk * dv
    st = qs.new_state(cq)
    st.widths.copy_(torch.from_numpy(widths))
    st.head_off.copy_(torch.from_numpy(off.view(np.int32)))
    S = torch.from_numpy(rng.standard_normal((2, 3, dk, dv)).astype(np.float32)).cuda()
    for call in (lambda: qs.qstate_pack(cq, S, st), lambda: qs.qstate_unpack(cq, st, S)):
        call()
        with pytest.raises(qs.QstateError):
            qs.qstate_check()
    qs.qstate_check()
