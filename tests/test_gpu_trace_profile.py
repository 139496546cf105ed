"""The cycle totals behind a trace: the unit scheduler's, never zeros."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1906_03113_gb300 as abfs  # noqa: E402


def test_cycle_totals_come_from_the_scheduler_only():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    abfs.build()
    torch.cuda.set_device(0)
    g = synth.rmat(14, 8.0, seed=2)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    s = int(np.argmax(g.degrees()))
    _, _, trace = abfs.run_trace(G, s)
    assert trace[0]["kind"] == "start" and trace[-1]["kind"] == "end"
    _, _, trace = abfs.run_trace(G, s, params=abfs.default_params(ctas_per_sm=1))
    assert trace[-2]["kind"] == "end" and trace[-1]["kind"] == "profile"
    assert trace[-1]["expand"] + trace[-1]["narrow_expand"] > 0
    G.destroy()
