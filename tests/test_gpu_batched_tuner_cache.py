"""A schedule that an older kernel's timings put into the tuner's cache is not taken."""
import json
import re

import numpy as np
import pytest

import workloads as W
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def test_schedules_of_older_kernels_are_timed_again(tmp_path):
    torch, cb = need_gpu()
    mats = [W.convdiff3d(s) for s in (6, 9, 12)]
    b = torch.from_numpy(np.concatenate([W.random_vector(A.n, 1) for A in mats])).cuda()
    x = torch.zeros_like(b)
    new, old = tmp_path / "new.jsonl", tmp_path / "old.jsonl"
    with cb.BatchedSolver(mats, restart=20, fmt="f32") as s:
        s.tune(b, x, tol=1e-8, cache_path=str(new))
        line = json.loads(new.read_text())
        # the key as it was written before it named the kernels' version
        line.update(key=re.sub(r"\|k\d+$", "", line["key"]), cluster=2, split_rows=4097, lanes=8)
        old.write_text(json.dumps(line) + "\n")
        assert s.tune(b, x, tol=1e-8, cache_path=str(old))[1] != 4097
        assert len(old.read_text().splitlines()) == 2        # timed and stored
        again = s.tune(b, x, tol=1e-8, cache_path=str(old))
        assert again[1] != 4097 and len(old.read_text().splitlines()) == 2   # and taken from then on
