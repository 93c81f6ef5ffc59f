"""The head unit's write-back at each way a lane's codes lie in a row (parts of words; one or two whole bytes
for 4 and 8 bits), each state shape, and intervals of one, several and an uneven number of tokens, whose
inputs are loaded a token ahead.  In lockstep with the oracle, under its bounds."""
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
