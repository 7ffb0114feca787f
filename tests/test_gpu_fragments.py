"""BITCOS from two tokens on: tiles decoded in tensor-core fragment order, one or two per warp.

Two tiles per warp are taken from 64 tiles per multiprocessor on.  The shapes lie on both sides of that line and where
the pairing can go wrong: an odd number of groups (the last warp of a row block has one tile), a single group, rows cut
into column blocks of odd width, a ragged last row block.  Against the oracle, within 1e-5 of sum|terms|.
"""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL = 1e-5


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_16338_b200 as m
    from paper_2609_16338_b200 import build
    build.build()
    m.load_library()
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check(y, y_ref, mag, what):
    yv = y.cpu().numpy().astype(np.float64)
    assert (np.abs(yv - y_ref) <= REL * mag).all(), what
    assert (yv[mag == 0] == 0).all(), what


@pytest.mark.parametrize("groups,above", [(1, True), (5, True), (5, False), (20, True), (39, True), (41, True), (57, True)])
def test_products_around_the_two_tile_line(bc, groups, above):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = -(-64 * sms // groups) - (0 if above else 1)          # row blocks: the line is 64 tiles per multiprocessor
    M, K = 32 * blocks - 5, 128 * groups
    W, S = datagen.trits(groups, M, K, 0.4219), datagen.scales(groups, M, K)
    Wd, ws = bc.bitcos_pack(W, S).to_device(), bc.make_workspace(M, K)
    for B in (2, 3, 8, 13):
        x, xs = datagen.activations(groups + B, B, K)
        _, y_ref, mag = oracle.gemv_dense(W, S, x, xs)
        y, _ = bc.bitcos_gemv(Wd, dev(x), dev(xs), workspace=ws)
        check(y, y_ref, mag, (groups, B))
        y2 = torch.full_like(y, float("nan"))
        bc.bitcos_gemv_multi([(Wd, dev(x), dev(xs), y2, ws)])
        assert torch.equal(y, y2)
        # one scale per token and group: equal scales give the per-token product
        xg = np.repeat(xs[:, None], groups, axis=1)
        yg, _ = bc.bitcos_gemv_group_scales(Wd, dev(x), dev(xg), workspace=ws)
        check(yg, y_ref, mag, (groups, B, "group scales"))
    assert bc.workspace_status(ws) == 0


def test_bf16_activations_with_two_tiles_per_warp(bc):
    """Two tokens quantised inside the launch: the two tiles of a warp are two different groups."""
    M, K = 32 * 500 - 9, 128 * 21
    W, S = datagen.trits(3, M, K, 0.4219), datagen.scales(3, M, K)
    Wd, ws = bc.bitcos_pack(W, S).to_device(), bc.make_workspace(M, K)
    xb = dev(datagen.activations_bf16(5, 2, K).view(np.int16)).view(torch.bfloat16)
    xq, xg = bc.bitcos_quantize_activations(xb)
    want, _ = bc.bitcos_gemv_group_scales(Wd, xq, xg, workspace=ws)
    got, _ = bc.bitcos_gemv_bf16(Wd, xb, workspace=ws)
    assert torch.equal(got, want)


@pytest.mark.parametrize("groups,blocks", [(1, 9472), (5, 1895), (41, 232), (54, 80), (3, 1)])
def test_16_bit_variant(bc, groups, blocks):
    """Weights +-1 in fragment order against bf16 activations, one and two tiles per warp, four and eight columns; the
    bound is the one of the variant's own tests ((128 + 200) fp32 additions of exact products)."""
    M, K = 32 * blocks - 3, 128 * groups
    W, S = datagen.trits(groups + 7, M, K, 0.4711), datagen.scales(groups, M, K)
    Wd, ws = bc.bitcos_pack(W, S).to_device(), bc.make_workspace(M, K)
    for B in (1, 4, 5, 8):
        bits = datagen.activations_bf16(groups + B, B, K)
        y_ref, mag = oracle.gemv_dense_blend(W, S, datagen.bf16_bits_to_f32(bits))
        y = bc.bitcos_gemv_blend_bf16(Wd, dev(bits.view(np.int16)).view(torch.bfloat16), workspace=ws)
        err = np.abs(y.cpu().numpy().astype(np.float64) - y_ref)
        assert (err <= 2e-5 * mag).all(), (groups, B)
    assert bc.workspace_status(ws) == 0


@pytest.mark.parametrize("groups", [9, 10, 11, 13, 15, 16, 17, 18, 19, 20, 36, 38])
def test_partial_sums_in_full_and_guarded_batches(bc, groups):
    """The epilogue adds a row block's sums ten at a time, with a second batch for more than ten; rows of such numbers of
    tiles (36 and 38: two column blocks of 18 and 19), all three formats, four to sixteen tokens."""
    M, K = 32 * 7 - 3, 128 * groups
    W, S = datagen.trits(700 + groups, M, K, 0.42), datagen.scales(700 + groups, M, K)
    ws, tiled = bc.make_workspace(M, K), bc.scales_tile(S, M, K)
    calls = ((bc.bitcos_gemv, bc.bitcos_pack(W, S).to_device()), (bc.trit5_gemv, bc.plain_to_device(bc.trit5_pack(W), tiled, M, K)),
             (bc.bit2_gemv, bc.plain_to_device(bc.bit2_pack(W), tiled, M, K)))
    for B in (4, 7, 16):
        x, xs = datagen.activations(700 + groups + B, B, K)
        _, y_ref, mag = oracle.gemv_dense(W, S, x, xs)
        for call, Wd in calls:
            y, _ = call(Wd, dev(x), dev(xs), workspace=ws)
            check(y, y_ref, mag, (call.__name__, groups, B))
    assert bc.workspace_status(ws) == 0
