"""What ptadd_batch_get_info reports of the work list, and what the tuner does where its candidates do not
differ: an FP64 batch cuts its own tiles and chunks."""

import json

import numpy as np
import pytest

from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MAT = W.Material().as_tuple()


def items(batch, tile, chunk):
    """Work items of tiles of `tile` targets and chunks of `chunk` sources."""
    total = 0
    for r in range(batch.R):
        nt = batch.realisation(r)
        nxt = np.concatenate([np.roll(np.arange(a, b), -1) for a, b in zip(nt.loop_off, nt.loop_off[1:])])
        targets = int(np.count_nonzero(~((nt.pinned != 0) & (nt.pinned[nxt] != 0))))
        total += -(-targets // tile) * -(-nt.n_nodes // chunk)
    return total


@pytest.mark.parametrize("R,loops", [(2, 1), (9, 16), (5, 40)])
def test_reported_tiles_and_chunks_give_the_work_items(R, loops):
    nets = [W.loop_ensemble(40 + r, loops, 0.8e-6, np.zeros(6)) for r in range(R)]
    batch = W.batch_from_networks(nets)
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.batch_set(batch)
        info = c.batch_info()
        assert info["tile_targets"] == 32
        assert info["work_items"] == items(batch, 32, info["chunk_sources"])
        c.set_precision(ptadd.PTADD_MIXED)
        c.batch_advance(1, 5e-13)
        info = c.batch_info()
        assert info["tile_targets"] in (64, 128)
        assert info["work_items"] == items(batch, info["tile_targets"], info["chunk_sources"])


def test_tuning_a_small_fp64_batch_keeps_the_default(tmp_path):
    """All six candidates are one work list here: no choice by the noise of their times."""
    nets = [W.loop_ensemble(80 + r, 6, 0.6e-6, np.zeros(6)) for r in range(4)]
    for k in range(4):
        cache = str(tmp_path / ("tune%d.jsonl" % k))
        with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
            c.batch_set(W.batch_from_networks(nets))
            before = c.batch_info()
            c.batch_autotune(cache, force=True)
            after = c.batch_info()
        assert after["tuned"] == 1
        assert {k: v for k, v in after.items() if k != "tuned"} == {k: v for k, v in before.items() if k != "tuned"}
        entries = [json.loads(line) for line in open(cache)]
        assert [(e["tpb"], e["chunk"]) for e in entries] == [(64, 2048)]
