"""Launches that begin while the one before them ends: a write-back must see all that earlier work on
its stream wrote, whatever that was (a torch kernel writing its inputs, another step, a copy), and the
same under graph capture.  Compared with the same calls with a synchronisation after each."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402

CASES = [("tiny_kda", dict(T=40), {}), ("kda_decode", dict(B=2, H=4, T=24, gate_bits=0), {}),
         ("gdn_decode", dict(B=2, H=4, T=24), {}), ("kda_prefill", dict(B=1, H=4, T=8 * 32, C=32), dict(interval_form=1)),
         ("kda_decode", dict(B=1, H=2, T=24, gate_bits=0), dict(alloc_mode=1))]


@pytest.mark.parametrize("name,size,over", CASES, ids=lambda v: str(v))
@pytest.mark.parametrize("capture", [False, True])
def test_steps_see_the_work_before_them(qs, name, size, over, capture):
    w = synth.scaled(synth.WORKLOADS[name], **size)
    cfg = qs.Config.from_workload(w, **over)
    src = synth.device_inputs(w)
    out = []
    for sync in (True, False):
        x = {n: torch.zeros_like(t) for n, t in src.items()}
        X = qs.Inputs(x["q"], x["k"], x["v"], x["s"], None, None, x.get("beta"), w.T)
        A, B, st = qs.new_state(cfg), qs.new_state(cfg), qs.new_stats(cfg)
        o = torch.zeros((w.B, w.T, w.H, w.dv), device="cuda")
        copy = torch.zeros_like(o)

        def steps(wait):
            a, b = A, B
            qs.qstate_init(cfg, a, b)
            for i, t in enumerate(range(0, w.T, cfg.C)):
                e = min(t + cfg.C, w.T)
                for n in x:   # the token's inputs, written just before on the same stream
                    torch.mul(src[n][:, t:e], 1.0, out=x[n][:, t:e]) if x[n][:, t:e].is_contiguous() else x[n][:, t:e].copy_(src[n][:, t:e])
                if wait:
                    torch.cuda.synchronize()
                qs.qstate_step(cfg, a, b, X, t, e, i, o, st)
                if wait:
                    torch.cuda.synchronize()
                copy[:, t:e].copy_(o[:, t:e])   # read right after
                for n in x:
                    x[n][:, t:e].fill_(float("nan"))   # and overwritten
                if wait:
                    torch.cuda.synchronize()
                a, b = b, a
            return a

        if sync or not capture:
            fin = steps(sync)
        else:
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s):
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s):
                    fin = steps(False)
                for _ in range(2):   # a replay starts from qstate_init again
                    g.replay()
            torch.cuda.current_stream().wait_stream(s)
        qs.qstate_check()
        out.append([t.cpu().view(torch.int32) if t.dtype == torch.float32 else t.cpu()
                    for t in (copy, fin.payload, fin.scales, fin.widths, fin.head_off, fin.fidx, st.ema_s, st.ema_r)])
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("name,size,over", [("kda_decode", dict(B=4, H=4, T=12, gate_bits=0), {}),
                                            ("gdn_decode", dict(B=4, H=16, T=12), {}),
                                            ("kda_prefill", dict(B=4, H=2, T=6 * 32, C=32), dict(interval_form=1))],
                         ids=lambda v: str(v))
@pytest.mark.parametrize("capture", [False, True])
def test_steps_after_a_partitioned_scan(qs, name, size, over, capture):
    """A launch that may begin early behind the join of several streams: a scan in partitions, then steps and
    another scan, against the same in one partition with a synchronisation after each call."""
    w = synth.scaled(synth.WORKLOADS[name], **size)
    cfg = qs.Config.from_workload(w, **over)
    x = synth.device_inputs(w)
    X = qs.Inputs(x["q"], x["k"], x["v"], x["s"], None, None, x.get("beta"), w.T)
    C, third = cfg.C, w.T // 3
    out = []
    for sync in (True, False):
        A, B, st = qs.new_state(cfg), qs.new_state(cfg), qs.new_stats(cfg)
        o = torch.zeros((w.B, w.T, w.H, w.dv), device="cuda")

        def calls():
            a, b = A, B
            wait = torch.cuda.synchronize if sync else lambda: None
            qs.qstate_init(cfg, a, b)
            wi = 0
            for lo, scan in ((0, True), (third, False), (2 * third, True)):
                hi = lo + third
                if scan:
                    if qs.qstate_scan(cfg, a, b, X, lo, hi, wi, o, st):
                        a, b = b, a
                    wi += third // C
                    wait()
                else:
                    for t in range(lo, hi, C):
                        qs.qstate_step(cfg, a, b, X, t, t + C, wi, o, st)
                        wi += 1
                        a, b = b, a
                        wait()
            return a

        qs.qstate_set_scan_partitions(1 if sync else 0)
        try:
            if not sync:
                assert qs.qstate_scan_partition_count(cfg, X, st) > 1
            if sync or not capture:
                fin = calls()
            else:
                s = torch.cuda.Stream()
                s.wait_stream(torch.cuda.current_stream())
                with torch.cuda.stream(s):
                    calls()   # the library's streams are made outside the capture
                    torch.cuda.synchronize()
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=s):
                        fin = calls()
                    for _ in range(2):
                        g.replay()
                torch.cuda.current_stream().wait_stream(s)
        finally:
            qs.qstate_set_scan_partitions(0)
        qs.qstate_check()
        out.append([t.cpu().view(torch.int32) if t.dtype == torch.float32 else t.cpu()
                    for t in (o, fin.payload, fin.scales, fin.widths, fin.head_off, fin.fidx, st.ema_s, st.ema_r)])
    for a, b in zip(*out):
        assert torch.equal(a, b)
