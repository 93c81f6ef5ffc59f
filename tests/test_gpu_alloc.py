"""The allocation kernel at the edges of its launch rule (units per thread, threads, series, ranked
list against histograms), bit for bit against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (B, H, dk, dv, head unit, heads per group): units on both sides of 1024, 2048, 4096 and 8192, up to
# the largest; batches on both sides of 32
SHAPES = [(2, 1, 64, 64, 0, 1), (1, 8, 128, 64, 0, 2), (1, 9, 128, 128, 0, 3), (31, 17, 128, 128, 0, 1),
          (33, 17, 128, 128, 0, 1), (32, 32, 128, 128, 0, 32), (2, 33, 128, 64, 0, 1), (2, 64, 128, 64, 0, 8),
          (1, 65, 128, 128, 0, 5), (1, 128, 128, 128, 0, 1), (1, 256, 64, 64, 0, 4), (3, 1, 128, 128, 1, 1),
          (2, 37, 128, 128, 1, 1), (1, 1024, 64, 64, 1, 1)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("stats", ["spread", "large_erasure", "levels", "tied", "null", "misaligned"])
def test_alloc_launch_rule(qs, orc, shape, stats):
    B, H, dk, dv, head, group = shape
    kw = dict(B=B, H=H, dk=dk, dv=dv, decay_kind=1 if head else 0, unit_kind=head, group_heads=1 if head else group,
              bmin=1, bmax=8)
    cq, co = qs.Config(bbar_num=3, bbar_den=1, **kw), orc.Cfg(bbar_num=3, **kw)
    n = B * cq.units
    rng = np.random.default_rng(n)
    ms = rng.uniform(0.02, 0.7, n).astype(np.float32)
    mr = rng.uniform(0, 0.02 if stats != "large_erasure" else 2.5, n).astype(np.float32)
    R = np.exp(rng.normal(0, 1, n)).astype(np.float32)
    if stats == "levels":          # several hundred units share each weight: the tied ones by index
        ms, mr, R = (np.round(a * 2).astype(np.float32) / 2 + np.float32(0.25) for a in (ms, mr, R))
    elif stats == "tied":
        ms[:], mr[:], R[:] = 0.25, 0.0, 1.0
    elif stats == "null":          # most weights are null: the threshold lies among them
        ms[rng.random(n) < 0.9] = 1.0
    pad = 1 if stats == "misaligned" else 0
    put = lambda a: torch.from_numpy(np.concatenate([np.zeros(pad, a.dtype), a])).cuda()[pad:]  # noqa: E731
    st = qs.Stats(put(ms), put(mr), put(R))
    widths, off = put(np.zeros(n, np.uint8)), torch.zeros(B * H, dtype=torch.int32, device="cuda")
    qs.qstate_alloc_bits(cq, st, widths, off)
    qs.qstate_check()
    wref, oref = orc.alloc(co, ms, mr, R)
    assert np.array_equal(widths.cpu().numpy(), wref)
    assert np.array_equal(off.cpu().numpy().view(np.uint32), oref)


@pytest.mark.parametrize("shape", [(2, 1, 64, 64, 0, 1), (2, 33, 128, 64, 0, 1), (1, 128, 128, 128, 0, 1), (2, 37, 128, 128, 1, 1)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("kind", [0, 2, 6, 7])
def test_alloc_statistics_beyond_range(qs, orc, shape, kind):
    """Erasure statistics that overflowed, or are NaN: those units weigh nothing (NaN: as without erasure)."""
    B, H, dk, dv, head, group = shape
    kw = dict(B=B, H=H, dk=dk, dv=dv, decay_kind=head, unit_kind=head, group_heads=group, bmin=1, bmax=8, weight_kind=kind)
    cq, co = qs.Config(bbar_num=3, bbar_den=1, **kw), orc.Cfg(bbar_num=3, **kw)
    n = B * cq.units
    rng = np.random.default_rng(n + kind)
    ms, mr = rng.uniform(0.02, 0.7, n).astype(np.float32), rng.uniform(0, 0.02, n).astype(np.float32)
    R = np.exp(rng.normal(0, 1, n)).astype(np.float32)
    for v in (np.inf, -np.inf, np.nan, np.finfo(np.float32).max, 1e20, 89.0, 88.0):
        mr[rng.choice(n, max(1, n // 50), replace=False)] = v
    put = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    widths, off = put(np.zeros(n, np.uint8)), torch.zeros(B * H, dtype=torch.int32, device="cuda")
    qs.qstate_alloc_bits(cq, qs.Stats(put(ms), put(mr), put(R)), widths, off)
    qs.qstate_check()
    wref, oref = orc.alloc(co, ms, mr, R)
    assert np.array_equal(widths.cpu().numpy(), wref)
    assert np.array_equal(off.cpu().numpy().view(np.uint32), oref)


@pytest.mark.parametrize("shape", [(2, 33, 128, 64, 0, 1), (1, 65, 64, 64, 0, 5), (1, 65, 128, 128, 0, 5), (1, 128, 128, 128, 0, 1),
                                   (2, 65, 128, 128, 1, 1), (1, 1024, 64, 64, 1, 1)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("kind", [1, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("pad", [0, 1])
def test_alloc_other_weights(qs, orc, shape, kind, pad):
    """The other weights at every number of units per thread, aligned and not; heads above 64, whose offsets
    are summed by a warp for each 32."""
    B, H, dk, dv, head, group = shape
    kw = dict(B=B, H=H, dk=dk, dv=dv, decay_kind=head, unit_kind=head, group_heads=group, bmin=1, bmax=8,
              weight_kind=kind, C=13)
    cq, co = qs.Config(bbar_num=3, bbar_den=1, **kw), orc.Cfg(bbar_num=3, **kw)
    n = B * cq.units
    rng = np.random.default_rng(n + kind)
    ms, mr = rng.uniform(0.02, 0.7, n).astype(np.float32), rng.uniform(0, 0.3, n).astype(np.float32)
    R = np.exp(rng.normal(0, 1, n)).astype(np.float32)
    put = lambda a: torch.from_numpy(np.concatenate([np.zeros(pad, a.dtype), a])).cuda()[pad:]  # noqa: E731
    widths, off = put(np.zeros(n, np.uint8)), torch.zeros(B * H, dtype=torch.int32, device="cuda")
    qs.qstate_alloc_bits(cq, qs.Stats(put(ms), put(mr), put(R)), widths, off)
    qs.qstate_check()
    wref, oref = orc.alloc(co, ms, mr, R)
    assert np.array_equal(widths.cpu().numpy(), wref)
    assert np.array_equal(off.cpu().numpy().view(np.uint32), oref)
