"""The drafters' draws at a low temperature where two race blocks with different
maxima nearly tie: the log-domain keys must not lose what the products of the
maxima and log2(e) / tau are rounded by (near_ties.py)."""
import numpy as np
import pytest
import torch

import near_ties
from test_gpu_draft import run_draft, run_oracle_draft
from test_gpu_markov import run_markov

pytestmark = pytest.mark.gpu


def _case(V, a, b, limit=None):
    ids, winner = near_ties.find(a, b)
    ids, winner = ids[:limit], winner[:limit]
    assert len(ids) > 20 and len(set(winner.tolist())) == 2
    logits = torch.as_tensor(near_ties.row(V, a, b)).to(torch.bfloat16).expand(len(ids), 1, V).contiguous()
    i64 = lambda x: torch.as_tensor(np.asarray(x, np.int64))
    return logits, (i64([near_ties.SEED] * len(ids)), i64(ids), i64([near_ties.POSITION] * len(ids))), winner


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V,a,b", [(4096, 1, 9), (4096, 14, 3), (25000, 90, 2)])
def test_draft(dtype, V, a, b):
    logits, requests, winner = _case(V, a, b)
    want = run_oracle_draft(logits, float(near_ties.TAU), *requests)["z"][:, 0]
    assert (want // 256).tolist() == winner.tolist()
    got = run_draft(logits.to(dtype), float(near_ties.TAU), *requests)
    assert got["status"] == 0
    assert (got["z"][:, 0] // 256).tolist() == winner.tolist()


@pytest.mark.parametrize("V,a,b", [(1024, 0, 2), (4096, 14, 3), (5000, 18, 2)])
def test_markov(V, a, b):
    """W1 = 0, so that the logits are U exactly."""
    logits, requests, winner = _case(V, a, b, limit=128)
    B = len(winner)
    zero = torch.zeros((V, 64), dtype=torch.bfloat16)
    got = run_markov(logits, zero, zero.t(), torch.zeros(B, dtype=torch.int32), float(near_ties.TAU), *requests)
    assert got["status"] == 0
    assert (got["z"][:, 0] // 256).tolist() == winner.tolist()
