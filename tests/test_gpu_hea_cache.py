"""An autotuner file of before the HEA's own sweep does not keep its boundaries on the tile passes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,prec,name,entry", [(7, 1, "fp32", "12 4 256 0"), (8, 1, "fp32", "12 5 256 4"),
                                               (7, 0, "fp64", "99 0 0 0"), (8, 0, "fp64", "13 4 256 0")])
def test_stale_entry_is_replaced(fp, L, prec, name, entry, tmp_path, monkeypatch):
    import torch
    cache = tmp_path / "tune.txt"
    line = f"{torch.cuda.get_device_name(0)} n=20 l={L} {name} hea|"
    cache.write_text(line + entry + "\n")
    monkeypatch.setenv("FP_AUTOTUNE_CACHE", str(cache))
    got = []
    for _ in range(2):      # the second ensemble finds the new entry
        ens = fp.Ensemble(fp.HEA, 20, L, L, seed=4)
        got.append(ens.trace_batch(0, 5, prec)[0])
        assert ens.brick_variant(L, prec)[3] == 5
        ens.close()
    assert np.array_equal(got[0], got[1])
    lines = [x for x in cache.read_text().splitlines() if x.startswith(line)]
    assert len(lines) == 2 and lines[1].endswith(" 5"), lines
