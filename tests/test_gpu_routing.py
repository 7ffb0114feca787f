"""bitcos_group_pairs_device against the host's stable grouping: one pair, warps and blocks of pairs with remainders, the
largest list, every expert the same, expert ids out of range (dropped; the rest of the lists filled)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_16338_b200 as m
    from paper_2609_16338_b200 import build
    build.build()
    m.load_library()
    return m


@pytest.mark.parametrize("pairs,experts,bad", [(1, 1, 0), (1, 1024, 0), (31, 3, 0), (33, 128, 5), (64, 128, 0), (257, 5, 40), (1000, 1024, 0),
                                               (4096, 1024, 0), (4095, 1, 0), (4096, 7, 4096), (96, 128, 31)])
def test_pairs_grouped_as_on_the_host(bc, pairs, experts, bad):
    rng = np.random.default_rng(pairs + experts)
    pe = rng.integers(0, experts, pairs).astype(np.int32)
    pe[rng.permutation(pairs)[:bad]] = rng.choice(np.array([-1, experts, 1 << 20, -(1 << 31)], np.int64), bad).astype(np.int32)
    pr = rng.integers(0, 1 << 20, pairs).astype(np.int32)
    ge, gb, xr, order, ng = (t.cpu().numpy() for t in bc.bitcos_group_pairs_device(torch.from_numpy(pe).cuda(), torch.from_numpy(pr).cuda(), experts))
    kept = np.flatnonzero((pe >= 0) & (pe < experts))
    want = kept[np.argsort(pe[kept], kind="stable")]
    n, cap = len(want), min(pairs, experts)
    ids, first = np.unique(pe[want], return_index=True)
    assert int(ng[0]) == len(ids)
    assert np.array_equal(order, np.concatenate([want, np.full(pairs - n, -1)]))
    assert np.array_equal(xr, np.concatenate([pr[want], np.zeros(pairs - n, np.int32)]))
    assert np.array_equal(ge, np.concatenate([ids, np.zeros(cap - len(ids), np.int32)]))
    assert np.array_equal(gb, np.concatenate([first, [n], np.zeros(cap - len(ids), np.int32)]))
