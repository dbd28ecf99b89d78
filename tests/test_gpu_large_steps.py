"""Steps of more than 2^21 and more than 2^23 occurrences against the CPU oracle
on tracked rows: the sort tiles, the scan and the lane-group limit of the row
kernels change there (needs a GPU)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2205_11048_gb300 import binding as B
from paper_2205_11048_gb300 import workload as W
from tests import _harness as H

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

# kept occurrences of the tracked rows: both sides of the row kernels' limits
# (4; 32 up to 2^23 occurrences, 64 above), and rows of one and several chunks
COUNTS = [1, 2, 3, 4, 5, 6, 31, 32, 33, 34, 63, 64, 65, 66, 127, 128, 129, 1000, 6000]
SHAPE = [(600_000, 4, 0), (90_000, 4, 0), (400_000, 6, 0)]  # rows, width, optimizer
SCAN_CACHE_BYTES, SEG_TABLE_BYTES = 20 * 1024, 96  # what the scan keeps in shared memory


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n", [(1 << 21) + 5001, (1 << 23) + 5001])
@pytest.mark.parametrize("M", [5, 700])
@pytest.mark.parametrize("rule", [dict(iota=0), dict(iota=1, decay=1, lam=0.5)])
def test_large_steps_against_the_oracle(n, M, rule):
    """Three tables whose borders fall inside a scan tile, ragged messages (so
    many that the scan's lookups stay in global memory, or few), a step of fresh
    ones and one with stale ones, dropped (iota 0) or halved (decay)."""
    T = len(SHAPE)
    lookups = T * SEG_TABLE_BYTES + 4 * M + 8 * T * M + 4 * T * (M + 1)
    assert (lookups > SCAN_CACHE_BYTES) == (M > 100)
    D = 8
    opts = [B.opt_desc(kind, 0.01) for _, _, kind in SHAPE]
    rng = np.random.default_rng(n + M)
    part = [int(0.45 * n), int(0.1 * n)]
    part.append(n - sum(part))
    assert part[0] % 2048 and (part[0] + part[1]) % 2048
    track = []
    for rows, _, _ in SHAPE:
        others = rng.choice(np.arange(len(COUNTS), rows), 300, replace=False)
        track.append(np.unique(np.concatenate([np.arange(len(COUNTS)), others])).astype(np.int64))
    g = B.GBA([(r, d, 0, part[t], opts[t]) for t, (r, d, _) in enumerate(SHAPE)], D, B.opt_desc(0, 0.01),
              M, M, seed=9, **rule)
    g.set_debug(True)
    orc = O.OracleGBA([O.TableSpec(r, d, O.OptSpec(kind, 0.01), 0) for r, d, kind in SHAPE], D,
                      O.OptSpec(0, 0.01), M, seed=9, track_rows=track, track_dense=None, **rule)
    for k in range(2):
        gen = torch.Generator(device="cuda").manual_seed(n + M + k)
        ids, grads, cuts = [], [], []
        for t, (rows, d, _) in enumerate(SHAPE):
            some = np.repeat(np.arange(len(COUNTS)), COUNTS)
            rest = rng.integers(len(COUNTS), rows, part[t] - len(some))
            ids.append(rng.permutation(np.concatenate([some, rest])).astype(np.int64))
            grads.append(torch.randn(part[t], d, generator=gen, device="cuda") * 0.01)
            cuts.append(np.concatenate([[0], np.sort(rng.integers(0, part[t] + 1, M - 1)), [part[t]]]))
        dev = [torch.as_tensor(i, device="cuda") for i in ids]
        seen = [np.nonzero(np.isin(i, tr))[0] for i, tr in zip(ids, track)]
        seen_grads = [x[torch.as_tensor(s, device="cuda")].cpu().numpy() for x, s in zip(grads, seen)]
        dense = torch.randn(M, D, generator=gen, device="cuda") * 0.01
        dense_host = dense.cpu().numpy()
        tokens = [k - int(k > 0 and m % 3 == 1) for m in range(M)]
        torch.cuda.synchronize()
        for m in range(M):
            of = [(int(c[m]), int(c[m + 1])) for c in cuts]
            g.push_ref(tokens[m], [dev[t][a:b] for t, (a, b) in enumerate(of)],
                       [grads[t][a:b] for t, (a, b) in enumerate(of)], dense[m], 1)
            mine = [slice(*np.searchsorted(seen[t], [a, b])) for t, (a, b) in enumerate(of)]
            orc.push(O.Message(tokens[m], 1, [ids[t][seen[t][s]] for t, s in enumerate(mine)],
                               [seen_grads[t][s] for t, s in enumerate(mine)], dense_host[m]))
        assert g.try_apply() == 1 and orc.try_apply() == 1
        g.sync()
        H.compare_segments(g, orc, False)
        H.compare_state(g, orc, H.TOL_ONE_STEP)
        if k == 0:
            t_g, r_g, _, kept_g = g.segments()
            for t in range(T):
                assert kept_g[t_g == t][:len(COUNTS)].tolist() == COUNTS
                assert r_g[t_g == t][:len(COUNTS)].tolist() == list(range(len(COUNTS)))
    assert g.stats()["occurrences"] == 2 * n
    g.close()
