"""Replays of one batch give the same energies bit for bit, whichever block takes a chunk of rays."""
import pytest

import synth
from tests.test_batch_gpu import _fields, _make, _tracers, torch  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1])
def test_energies_repeat(torch, kind):  # noqa: F811
    from paper_1001_3301_gb300 import Batch
    ws = _make(synth.batch_specs(12))
    trs = _tracers(ws)
    b = Batch(trs)
    assert b.tuning()[0] == 1
    if kind == 0:
        b.set_tuning(0, 8, 4)
    f = _fields(torch, ws)
    first = None
    for _ in range(8):
        b.run(*f)
        e = [(x.e_abs, x.e_esc) for x in b.energy()]
        first = first or e
        assert e == first
    b.close()
