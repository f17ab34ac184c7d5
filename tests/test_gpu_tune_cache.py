"""Choices that were tuned for other kernels are not taken over from the cache."""
import json

import pytest
import torch

from paper_1511_07174_gb300 import api, batched

pytestmark = pytest.mark.gpu


def _write(path, entries):
    path.mkdir(exist_ok=True)
    (path / "autotune.json").write_text(json.dumps(entries))


def test_entries_of_other_kernels_are_ignored(tmp_path, monkeypatch):
    monkeypatch.setenv("GBLA_CACHE", str(tmp_path))
    name = torch.cuda.get_device_name("cuda")
    g = torch.Generator().manual_seed(0)
    As = [torch.rand((n, n), generator=g, dtype=torch.float64) + n * torch.eye(n, dtype=torch.float64) for n in (5, 9)]
    bl = batched.BatchedLU(As)
    # the keys as they were, with choices that no candidate has
    _write(tmp_path, {"lu_nb|%s|200" % name: {"nb": 96}, "chol_nb|%s|200" % name: {"nb": 192},
                      "%s|lu|torch.float64|2|5|9|%d" % (name, (125 + 729) >> 20): {"threads": 512, "ctas_per_sm": 7}})
    assert api.tune_lu_nb(200, candidates=(128,)) == 128
    assert api.tune_chol_nb(200, candidates=(64,)) == 64
    bl.autotune(reps=1)
    assert (bl.threads, bl.ctas_per_sm) in batched.CANDIDATES
    # and the new ones are found again
    assert api.tune_lu_nb(200, candidates=(64,)) == 128
    cache = json.loads((tmp_path / "autotune.json").read_text())
    cache[bl.key()]["ctas_per_sm"] = 5
    _write(tmp_path, cache)
    assert bl.autotune()["ctas_per_sm"] == 5
