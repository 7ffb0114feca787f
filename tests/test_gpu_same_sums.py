"""One product, one order of its sums: the bits of y do not depend on how the product is launched.

Scales spread over many powers of two, so that no sum of a few of them is exact and any other order shows.
"""
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


def matrix(seed, M, K):
    """Trits on the device, and bf16 scales 1 .. 2 times 2^-6 .. 2^6."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((M, K), generator=gen, device="cuda")
    trits = (u >= 0.42).to(torch.int8) - 2 * (u >= 0.71).to(torch.int8)
    scales = torch.exp2(12 * torch.rand((M, K // 128), generator=gen, device="cuda") - 6).to(torch.bfloat16)
    return trits, scales


def activations(seed, B, K):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-127, 128, (B, K), generator=gen, device="cuda", dtype=torch.int8), 0.5 + torch.rand((B, K // 128), generator=gen, device="cuda")


def group_sums(trits, x):
    """int32 [batch, M, K / 128]; 128 products of at most 127 are exact in fp32."""
    G = trits.shape[1] // 128
    w = trits.view(-1, G, 128).permute(1, 0, 2).float()
    return torch.bmm(x.view(-1, G, 128).permute(1, 0, 2).float(), w.transpose(1, 2)).permute(1, 2, 0).round().to(torch.int32).contiguous()


@pytest.mark.parametrize("fmt,batches", [("bitcos", (1, 2, 3, 8, 16)), ("trit5", (1, 2)), ("bit2", (1, 2))])
@pytest.mark.parametrize("M,K", [(38016, 2560), (19200, 5120), (12795, 6912), (24000, 3456), (70, 384)])
def test_the_accumulator_dump_changes_nothing(bc, fmt, batches, M, K):
    """The kernels with several tiles per warp and the small launches: the same bits with and without the dump, the
    dump itself exact."""
    trits, scales = matrix(M + K, M, K)
    if fmt == "bitcos":
        W, call = bc.bitcos_pack_device(trits, scales), bc.bitcos_gemv
    else:
        pack, call = (bc.trit5_pack, bc.trit5_gemv) if fmt == "trit5" else (bc.bit2_pack, bc.bit2_gemv)
        W = bc.plain_to_device(pack(trits.cpu().numpy()), bc.scales_tile(scales.view(torch.int16).cpu().numpy().view(np.uint16), M, K), M, K)
    ws = bc.make_workspace(M, K)
    for B in batches:
        x, xg = activations(B, B, K)
        xs = xg[:, 0].contiguous()
        y, _ = call(W, x, xs, workspace=ws)
        y2, acc = call(W, x, xs, acc_debug=True, workspace=ws)
        assert torch.equal(acc, group_sums(trits, x)), B
        assert torch.equal(y, y2), B
        if fmt == "bitcos":
            y, _ = bc.bitcos_gemv_group_scales(W, x, xg, workspace=ws)
            y2, acc2 = bc.bitcos_gemv_group_scales(W, x, xg, acc_debug=True, workspace=ws)
            assert torch.equal(acc, acc2) and torch.equal(y, y2), B
    assert bc.workspace_status(ws) == 0


# Two to eight products that are launched with one tile per warp each and with several together, and one product above the
# line beside one below it: whole rows in an item, one and two column blocks of even and odd width, at the end
# of a row a run that is not full.
SETS = [[(8192, 2560)] * 2, [(4096, 384)] * 7 + [(9472 * 32, 128)], [(8190, 2432)] * 2, [(4096, 1792)] * 6, [(4096, 1664)] * 6,
        [(4096, 5120)] * 2, [(4100, 4992)] * 2, [(4600, 4736)] * 2, [(6144, 3456)] * 2, [(6144, 3200)] * 2, [(8192, 5120), (1024, 5120), (1024, 2688)]]


@pytest.mark.parametrize("shapes", SETS, ids=lambda s: "+".join("%dx%d" % mk for mk in s[:2]))
def test_several_products_in_a_launch_have_the_bits_of_each_alone(bc, shapes):
    Ws = [bc.bitcos_pack_device(*matrix(i, M, K)) for i, (M, K) in enumerate(shapes)]
    wss = [bc.make_workspace(M, K) for M, K in shapes]
    ys = {B: [torch.empty((B, M), device="cuda") for M, _ in shapes] for B in (1, 2, 3, 8, 16)}
    for B in ys:
        if B == 1 and max(K for _, K in shapes) > 2560:
            continue              # (one token: rows of more than 20 groups are cut by the launch's own plan)
        acts = {K: activations(K + B, B, K) for _, K in shapes}
        token = {K: xg[:, 0].contiguous() for K, (_, xg) in acts.items()}
        jobs = [(W, acts[W.K][0], token[W.K], y, ws) for W, y, ws in zip(Ws, ys[B], wss)]
        bc.bitcos_gemv_multi(jobs)
        for W, x, xs, y, ws in jobs:
            assert torch.equal(y, bc.bitcos_gemv(W, x, xs, workspace=ws)[0]), (B, W.M, W.K)
        if B <= 2 and max(K for _, K in shapes) <= 2560:
            phased = [torch.empty_like(y) for y in ys[B]]
            bc.bitcos_gemv_phased([j[:3] + (y, j[4]) for j, y in zip(jobs, phased)], [0] * len(jobs), bc.make_phased_sync())
            assert all(torch.equal(a, b) for a, b in zip(phased, ys[B])), B
        jobs = [(W, acts[W.K][0], acts[W.K][1], y, ws) for W, y, ws in zip(Ws, ys[B], wss)]
        bc.bitcos_gemv_multi_group_scales(jobs)
        for W, x, xg, y, ws in jobs:
            assert torch.equal(y, bc.bitcos_gemv_group_scales(W, x, xg, workspace=ws)[0]), (B, W.M, W.K, "group scales")
        if B <= 2:
            bf16 = {K: torch.randn((B, K), generator=torch.Generator(device="cuda").manual_seed(K), device="cuda").to(torch.bfloat16) for K in acts}
            bc.bitcos_gemv_multi_bf16([(W, bf16[W.K], None, y, ws) for W, y, ws in zip(Ws, ys[B], wss)])
            for W, y, ws in zip(Ws, ys[B], wss):
                assert torch.equal(y, bc.bitcos_gemv_bf16(W, bf16[W.K], workspace=ws)[0]), (B, W.M, W.K, "bf16")
    assert not any(bc.workspace_status(ws) for ws in wss)
