"""The range scan of large batches (the spellings that continue a pending
identifier, looked at inside it before the walk): the same masks and the same
counted work as in batches too small for it, and the same masks where more
spellings end the identifier than the row's list holds."""
import itertools

import numpy as np
import pytest

from tests.harness import GpuRun, oracle_masks, unpack
from workloads import configs

pytestmark = pytest.mark.gpu


def _counted(run):
    """Masks with the work counters on."""
    import torch
    work = torch.zeros(6, dtype=torch.int64, device="cuda")
    run.G.grid_spec_set_work_counters(run.spec.h, work)
    words, status = run.masks()
    run.G.grid_spec_set_work_counters(run.spec.h, None)
    torch.cuda.synchronize()
    assert not status.any()
    return words.copy(), work.cpu().tolist()


def _large(run, times):
    """The run's rows `times` times over, in one batch of the same spec."""
    big = object.__new__(GpuRun)
    big.__dict__.update(run.__dict__)
    big.B = run.B * times
    big.cfg = run.G.Configs(run.spec, big.B)
    big.status = run.torch.zeros(big.B, dtype=run.torch.int32, device="cuda")
    big.mask = run.torch.zeros((big.B, run.W), dtype=run.torch.int32, device="cuda")
    assert not big.build_configs(prefixes=[p for p in run.wl["prefixes"]] * times).any()
    return big


def test_large_batch_counts_the_same_work():
    run = GpuRun(configs.sql_admin(B=32))
    assert not run.build_configs().any()
    words, work = _counted(run)
    big_words, big_work = _counted(_large(run, 16))
    assert (big_words == np.tile(words, (16, 1))).all()
    assert all(x > 0 for x in work) and big_work == [16 * x for x in work]


def test_more_survivors_than_the_list_holds():
    wl = configs.sql_admin(B=4)
    letters = "abcdefghijklmnopqrstuvwxyz"
    tails = ["".join(x) for n in (1, 2, 3) for x in itertools.product(letters, repeat=n)]
    tokens = list(wl["tokens"])
    known = set(tokens)
    tokens += [t for t in ((x + " ").encode() for x in tails) if t not in known]
    lexicons = {"TABLE_NAME": ["t1"], "COLUMN_NAME": ["q"] + ["q" + x for x in tails]}
    byte = {t: i for i, t in reversed(list(enumerate(tokens))) if len(t) == 1}
    texts = ["select q", "select q from t1 where q", "select t1.q", "select q, qa"]
    wl = dict(wl, tokens=tokens, lexicons=lexicons, prefixes=[[byte[bytes([c])] for c in x.encode()] for x in texts])
    run = GpuRun(wl)
    assert not run.build_configs().any()
    assert run.spec.info()["verdict_classes"] < len(tails)
    words, work = _counted(run)
    big_words, big_work = _counted(_large(run, 80))
    assert (big_words == np.tile(words, (80, 1))).all()
    assert big_work[5] > 80 * work[5]  # the ranges were scanned, and walked because the lists overflowed
    rng = np.random.default_rng(5)
    ids = sorted(set(rng.integers(0, len(tokens), 400).tolist() + rng.integers(len(known), len(tokens), 400).tolist()))
    want = oracle_masks(wl, ids_per_row=[ids] * 4)
    bits = unpack(words, run.V)
    for b in range(4):
        assert (bits[b][ids] == np.asarray(want[b], np.uint8)).all()
