"""Tuning caches written before there were two engines."""
import json

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1906_03113_gb300 as abfs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    abfs.build()
    abfs.load()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("mode", [abfs.MODE_SUBMATRIX, abfs.MODE_PLAIN])
@pytest.mark.parametrize("batch", [False, True])
def test_old_lines_do_not_hide_the_new_engine(tmp_path, mode, batch):
    """A submatrix line without the engines' number is measured again and the new
    choice, appended, is the one that is found from then on.  The comparator has
    one engine: its old lines stand."""
    g = synth.er(3000, 6.0, seed=2)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    path = tmp_path / "tune.json"

    def tune():
        if batch:
            return abfs.batch_tune([G, G], [0, 1], mode, str(path))
        return abfs.tune(G, [0, 1], mode, str(path))

    tune()
    line = json.loads(path.read_text())
    line.pop("engines", None)
    line["tile"] = 992  # no candidate has it
    path.write_text(json.dumps(line, separators=(",", ":")) + "\n")
    best, _ = tune()
    if mode == abfs.MODE_PLAIN:
        assert best.tile == 992 and len(path.read_text().splitlines()) == 1
    else:
        assert best.tile != 992 and len(path.read_text().splitlines()) == 2
        again, _ = tune()
        assert again.as_dict() == best.as_dict() and len(path.read_text().splitlines()) == 2
    G.destroy()
