"""Routed products: the device's grouping of the pairs, and the grouped kernels' token parts.

bitcos_group_pairs_device against the host's stable grouping: one pair, warps and blocks of pairs with remainders, the
largest list, every expert the same, expert ids out of range (dropped; the rest of the lists filled)."""
import numpy as np
import pytest

import datagen
import oracle

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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("M,K,experts,most", [(768, 2048, 28, 16), (2048, 640, 32, 16), (2000, 768, 28, 8), (96, 640, 40, 16), (1000, 4096, 12, 13),
                                              (640, 1280, 30, 2), (64, 128, 8, 16)])
def test_groups_of_every_size(bc, M, K, experts, most):
    """Groups of 1 .. most tokens, rows in one piece (one flat list of items; more than eight tokens of a group run as two
    parts) and rows cut into column blocks (K = 4096), odd numbers of groups of 128.  One group with too many tokens, one
    that names no expert, an empty group: skipped, the two malformed ones with status 2."""
    Ws = [datagen.trits(60 + e % 5, M, K, 0.33) for e in range(experts)]
    Ss = [datagen.scales(60 + e, M, K) for e in range(experts)]
    E = bc.DeviceExperts([bc.bitcos_pack(Ws[e], Ss[e]).to_device() for e in range(experts)])
    rng = np.random.default_rng(M + K)
    sizes = np.concatenate([[1, most], rng.integers(1, most + 1, experts - 2)])
    x, xs = datagen.activations(M + K, 20, K)
    group_expert = rng.permutation(experts).astype(np.int32)
    begin = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    rows = rng.integers(0, 20, begin[-1]).astype(np.int32)
    _, y_ref, mag = oracle.grouped_dense(Ws, Ss, np.repeat(group_expert, sizes), rows, x, xs)
    ws = bc.make_workspace(M, K, copies=experts)
    y, _ = bc.bitcos_gemv_grouped(E, dev(group_expert), dev(begin), dev(rows), most, dev(x), dev(xs), workspace=ws)
    yv = y.cpu().numpy().astype(np.float64)
    assert (np.abs(yv - y_ref) <= 1e-5 * mag).all()
    assert bc.workspace_status(ws) == 0
    # group 3 takes all of group 4's pairs and more (too many), group 6 names no expert
    bad_begin, bad_expert = begin.copy(), group_expert.copy()
    bucket = next(b for b in (1, 2, 4, 8, 16) if b >= most)
    assert begin[6] - begin[3] > bucket
    bad_begin[4:6] = begin[6]
    bad_expert[6] = experts
    ws = bc.make_workspace(M, K, copies=experts)
    y2 = torch.full_like(y, 7.0)
    bc.bitcos_gemv_grouped(E, dev(bad_expert), dev(bad_begin), dev(rows), most, dev(x), dev(xs), y=y2, workspace=ws)
    want = y.clone()
    want[begin[6]:begin[7]] = 7.0
    want[begin[3]:begin[6]] = 7.0
    assert torch.equal(y2, want)
    assert bc.workspace_status(ws) == 2
