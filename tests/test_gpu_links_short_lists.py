"""The link kernel's batches at every size: a warp takes as many pairs (1 to 8)
as give each resident warp a batch, so the batch grows with the list.  One list
of pairs, walls and invalid pairs among them, repeated to lengths on either side
of the batch sizes and their remainders; each copy of a pair against the
oracle, and in arrays with and without room behind the list."""
import numpy as np
import pytest

import gen
import oracle
from test_gpu_links import MU, QBAR, lub  # noqa: F401  (lub: the module's fixture)

pytestmark = pytest.mark.gpu

RESIDENT = 152 * 5 * 4  # warps


@pytest.mark.parametrize("count", [1, 65, RESIDENT, RESIDENT + 1, 2 * RESIDENT + 7, 4 * RESIDENT + 1, 7 * RESIDENT,
                                   7 * RESIDENT + 1, 8 * RESIDENT + 13])
@pytest.mark.parametrize("room", [0, 30000])
def test_batches_grow_with_the_list(lub, count, room):
    import torch
    m = 65
    parts, dom, pi, pj = gen.pair_stream(m, seed=92, kind="mixed", gap_range=(0.02, 1.5))
    pi, pj = pi.copy(), pj.copy()
    bad = np.arange(m) % 5 == 3
    pj[bad] = np.where(np.arange(m)[bad] % 2 == 0, -1, pi[bad])
    at = np.arange(count) % m
    pl = lub.Pipeline(parts, dom, lub.default_params(), capacity=count + room)
    pl.set_pairs(pi[at], pj[at])
    F, T, nl = pl.links(QBAR)
    torch.cuda.synchronize()
    C = pl.cap
    F, T = F.cpu().numpy().reshape(3, C)[:, :count].T, T.cpu().numpy().reshape(6, C)[:, :count].T
    nl = nl[:count].cpu().numpy()
    ref = oracle.links(parts, dom, pi[~bad], pj[~bad], MU, QBAR)
    refF, refT, refn = np.zeros((m, 3)), np.zeros((m, 6)), np.zeros(m, np.int64)
    refF[~bad], refT[~bad], refn[~bad] = ref["F"], ref["T"], ref["links"]
    np.testing.assert_array_equal(nl, refn[at])
    np.testing.assert_allclose(F, refF[at], rtol=1e-9, atol=1e-12 * np.abs(refF).max())
    np.testing.assert_allclose(T, refT[at], rtol=1e-9, atol=1e-12 * np.abs(refT).max())
