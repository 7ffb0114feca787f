"""GPU parity for the device-side BITCOS packer: byte for byte the buffers the oracle builds from
the paper's layout (Section II-A: presence bitmap, compacted signs in the same order; entry
offsets per tile), and usable by the product as packed."""
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


def u32(t):
    return t.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("M,K,z", [(32, 128, 0.42), (1, 128, 0.5), (100, 384, 0.47), (640, 2560, 0.4219), (2560, 6912, 0.33),
                                   (4097, 1280, 0.42), (64, 256, 1.0), (64, 256, 0.0), (8192, 5120, 0.4711)])
def test_device_pack_matches_oracle_bytes(bc, M, K, z):
    W = datagen.trits(3000 + M, M, K, z)
    if z == 0.0:
        W[W == 0] = 1
    S = datagen.scales(3000 + M, M, K)
    ref = oracle.bitcos_pack(W)
    Wd = bc.bitcos_pack_device(torch.from_numpy(W).cuda(), torch.from_numpy(S.view(np.int16)).cuda())
    assert Wd.nnz == ref.nnz == bc.bitcos_count_nnz_device(torch.from_numpy(W).cuda())
    assert np.array_equal(u32(Wd.bitmap), ref.bitmap)
    n_tiles = oracle.num_tiles(M, K)
    off = u32(Wd.tile_off)
    assert np.array_equal(off[:n_tiles + 1], ref.tile_off) and not off[n_tiles + 1:].any()
    assert np.array_equal(Wd.tile_off_host, ref.tile_off)
    sg = u32(Wd.signs)
    n_words = (ref.nnz + 31) // 32
    assert np.array_equal(sg[:n_words], np.asarray(ref.signs, np.uint32)[:n_words]) and not sg[n_words:].any()
    assert np.array_equal(Wd.scales.cpu().numpy().view(np.uint16), oracle.scales_to_tile_order(S, M, K).reshape(-1))
    # and the library's host packer wrote the same bytes (sign slack included)
    host = bc.bitcos_pack(W, S)
    assert np.array_equal(sg, host.signs) and np.array_equal(off, host.tile_off_buf)


def test_device_packed_matrix_multiplies(bc):
    M, K, B = 2560, 2560, 3
    W, S = datagen.trits(3100, M, K, 0.4219), datagen.scales(3100, M, K)
    x, xs = datagen.activations(3100, B, K)
    acc_ref, y_ref, mag = oracle.gemv_dense(W, S, x, xs)
    Wd = bc.bitcos_pack_device(torch.from_numpy(W).cuda(), torch.from_numpy(S.view(np.int16)).cuda())
    y, acc = bc.bitcos_gemv(Wd, torch.from_numpy(x).cuda(), torch.from_numpy(xs).cuda(), acc_debug=True)
    torch.cuda.synchronize()
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    assert (np.abs(y.cpu().numpy().astype(np.float64) - y_ref) <= 1e-5 * mag).all()


def test_device_pack_error_codes(bc):
    M, K = 64, 256
    W = datagen.trits(3200, M, K, 0.4)
    S = datagen.scales(3200, M, K)
    bad = W.copy()
    bad[5, 17] = 2
    with pytest.raises(bc.BitcosError) as e:
        bc.bitcos_pack_device(torch.from_numpy(bad).cuda(), torch.from_numpy(S.view(np.int16)).cuda())
    assert e.value.status == 4
    bad[5, 17] = -2
    with pytest.raises(bc.BitcosError) as e:
        bc.bitcos_count_nnz_device(torch.from_numpy(bad).cuda())
    assert e.value.status == 4
    Sb = S.copy()
    Sb[3, 1] = 0x7F80                                  # +Inf
    with pytest.raises(bc.BitcosError) as e:
        bc.bitcos_pack_device(torch.from_numpy(W).cuda(), torch.from_numpy(Sb.view(np.int16)).cuda())
    assert e.value.status == 5
    Sb[3, 1] = 0x8000 | 0x3C00                         # negative
    with pytest.raises(bc.BitcosError) as e:
        bc.bitcos_pack_device(torch.from_numpy(W).cuda(), torch.from_numpy(Sb.view(np.int16)).cuda())
    assert e.value.status == 5
    with pytest.raises(bc.BitcosError) as e:
        bc.bitcos_pack_device(torch.zeros((4, 100), dtype=torch.int8, device="cuda"),
                              torch.zeros((4, 1), dtype=torch.int16, device="cuda"))
    assert e.value.status == 2


@pytest.mark.parametrize("M,K,z", [(32, 128 * 8191, 0.5), (32 * 4096, 256, 0.47), (32 * 4096 - 31, 256, 0.3), (3, 128 * 8193, 0.9)])
def test_device_pack_around_a_scan_pass(bc, M, K, z):
    """The entry offsets are scanned 8192 tiles at a time: one tile fewer, exactly as many, one more; and sign bits of
    a few non-zeros a tile, where several tiles share a word."""
    W, S = datagen.trits(3300 + M, M, K, z), datagen.scales(3300 + M, M, K)
    if z == 0.9:
        W[:, ::3] = 0
        W[1:] = 0
    Wd = bc.bitcos_pack_device(torch.from_numpy(W).cuda(), torch.from_numpy(S.view(np.int16)).cuda())
    host = bc.bitcos_pack(W, S)
    assert Wd.nnz == host.nnz
    assert np.array_equal(u32(Wd.bitmap), host.bitmap) and np.array_equal(u32(Wd.signs), host.signs)
    assert np.array_equal(u32(Wd.tile_off), host.tile_off_buf) and np.array_equal(Wd.tile_off_host, host.tile_off)
    assert np.array_equal(Wd.scales.cpu().numpy().view(np.uint16), host.scales)


def test_device_pack_into_a_vector_that_is_too_small(bc):
    """The C call with a sign vector one bit short, and exactly as large as needed; offsets to pageable memory."""
    import ctypes as C
    M, K = 96, 640
    W, S = datagen.trits(3400, M, K, 0.4), datagen.scales(3400, M, K)
    host = bc.bitcos_pack(W, S)
    L = bc.load_library()
    t, sc = torch.from_numpy(W).cuda(), torch.from_numpy(S.view(np.int16)).cuda()
    bitmap, off = torch.empty(host.bitmap.size, dtype=torch.int32, device="cuda"), torch.empty(host.tile_off_buf.size, dtype=torch.int32, device="cuda")
    signs, tiled = torch.empty(host.signs.size, dtype=torch.int32, device="cuda"), torch.empty(host.scales.size, dtype=torch.int16, device="cuda")
    scratch, off_host, nnz = torch.empty(256, dtype=torch.uint8, device="cuda"), np.zeros(host.tile_off_buf.size, np.uint32), C.c_uint64(0)
    for short, want in ((16, 6), (0, 0)):
        rc = L.bitcos_pack_device(t.data_ptr(), sc.data_ptr(), M, K, bitmap.data_ptr(), signs.data_ptr(), host.signs.nbytes - short,
                                  off.data_ptr(), tiled.data_ptr(), off_host.ctypes.data, C.byref(nnz), scratch.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
        assert rc == want
    assert nnz.value == host.nnz and np.array_equal(u32(signs), host.signs) and np.array_equal(off_host, host.tile_off_buf)


def test_device_pack_with_offsets_to_memory_that_is_pinned_in_part(bc):
    """The offsets go to the host by the packer's own stores only where all of the caller's buffer is mapped; a buffer of
    which one page is registered is left to the runtime's copy, which refuses it."""
    import ctypes as C
    import mmap
    M, K = 25600, 5120
    L = bc.load_library()
    gen = torch.Generator(device="cuda").manual_seed(5)
    t = torch.randint(-1, 2, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    sc = torch.full((M, K // 128), 0.5, device="cuda").to(torch.bfloat16)
    want = bc.bitcos_pack_device(t, sc)
    signs, off = torch.empty(M * K // 32 + 64, dtype=torch.int32, device="cuda"), torch.empty_like(want.tile_off)
    bitmap, tiled = torch.empty_like(want.bitmap), torch.empty_like(want.scales)
    scratch = torch.empty(256, dtype=torch.uint8, device="cuda")
    size = -(-4 * off.numel() // mmap.PAGESIZE) * mmap.PAGESIZE
    host = np.frombuffer(mmap.mmap(-1, size), dtype=np.uint32)
    rt = torch.cuda.cudart()
    for pinned, status in ((size, 0), (mmap.PAGESIZE, 8), (0, 0)):
        if pinned:
            assert int(rt.cudaHostRegister(host.ctypes.data, pinned, 0)) == 0
        host[:] = 0xFFFFFFFF
        rc = L.bitcos_pack_device(t.data_ptr(), sc.data_ptr(), M, K, bitmap.data_ptr(), signs.data_ptr(), 4 * signs.numel(), off.data_ptr(),
                                  tiled.data_ptr(), host.ctypes.data, None, scratch.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == status, pinned
        # (whatever happened, nothing of the call is still running)
        assert torch.cuda.current_stream().query(), pinned
        if status == 0:
            assert np.array_equal(host[:off.numel()].view(np.int32), want.tile_off.cpu().numpy()), pinned
            assert torch.equal(off, want.tile_off) and torch.equal(bitmap, want.bitmap), pinned
        if pinned:
            assert int(rt.cudaHostUnregister(host.ctypes.data)) == 0


@pytest.mark.parametrize("M,K", [(32 * 6143, 128), (32 * 6144, 128), (32 * 6145 - 7, 128), (32 * 1537, 512), (4097, 6144), (32 * 65121, 128),
                                 (32 * 180224, 128), (32 * 180225, 128)])
def test_device_pack_in_one_pass_and_in_three_kernels(bc, M, K):
    """Matrices on both sides of the lines between the packer's two ways (6144 and 180224 tiles), whole, against their
    upper and lower parts: the same bitmap and scales, offsets that go on where the upper part ends, the same sign bits."""
    gen = torch.Generator(device="cuda").manual_seed(M + K)
    t = torch.randint(-1, 2, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    top = M // 64 * 32
    # a multiple of 32 non-zeros above the cut, so that the sign words of the parts can be laid end to end
    extra = int((t[:top] != 0).sum()) % 32
    t.view(-1)[(t.view(-1)[:top * K] != 0).nonzero()[:extra, 0]] = 0
    sc = (0.01 + torch.rand((M, K // 128), generator=gen, device="cuda")).to(torch.bfloat16)
    whole, parts = bc.bitcos_pack_device(t, sc), [bc.bitcos_pack_device(a.contiguous(), b.contiguous()) for a, b in ((t[:top], sc[:top]), (t[top:], sc[top:]))]
    assert whole.nnz == parts[0].nnz + parts[1].nnz == int((t != 0).sum()) and parts[0].nnz % 32 == 0
    assert torch.equal(whole.bitmap, torch.cat([p.bitmap for p in parts])) and torch.equal(whole.scales, torch.cat([p.scales for p in parts]))
    first, words = parts[0].tile_off_host.size - 1, parts[0].nnz // 32
    off = np.concatenate([parts[0].tile_off_host[:-1], parts[1].tile_off_host + np.uint32(parts[0].nnz)])
    assert np.array_equal(whole.tile_off_host, off) and np.array_equal(u32(whole.tile_off)[:off.size], off) and first == top // 32 * (K // 128)
    last = (whole.nnz + 31) // 32
    assert torch.equal(whole.signs[:last], torch.cat([parts[0].signs[:words], parts[1].signs[:last - words]])) and not whole.signs[last:].any()
    del parts, off
    call = CPack(bc, t, sc)
    assert call.run() == (0, kernels(M, K), whole.nnz) and call.equals(whole)


def test_device_pack_in_one_pass_reports_what_is_wrong(bc):
    """A bad trit or scale in the last block of a large matrix, and the next call, which finds the shared state as it should be."""
    M, K = 8192, 5120
    gen = torch.Generator(device="cuda").manual_seed(9)
    t = torch.randint(-1, 2, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    sc = torch.full((M, K // 128), 0.5, device="cuda").to(torch.bfloat16)
    want = bc.bitcos_pack_device(t, sc)
    for value in (2, -2, 127, -128):
        bad = t.clone()
        bad[M - 1, K - 1] = value
        with pytest.raises(bc.BitcosError):
            bc.bitcos_pack_device(bad, sc)
    for value in (-1.0, float("inf"), float("nan")):
        bad = sc.clone()
        bad[M - 1, 0] = value
        with pytest.raises(bc.BitcosError):
            bc.bitcos_pack_device(t, bad)
    again = bc.bitcos_pack_device(t, sc)
    assert torch.equal(again.signs, want.signs) and torch.equal(again.tile_off, want.tile_off)


def test_device_pack_needs_no_free_chip(bc):
    """Kernels that stay on a few multiprocessors neither hold a pack up nor keep it from starting: it returns while they run."""
    M, K = 8192, 5120
    gen = torch.Generator(device="cuda").manual_seed(11)
    t = torch.randint(-1, 2, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    sc = torch.full((M, K // 128), 0.5, device="cuda").to(torch.bfloat16)
    want = [bc.bitcos_pack_device(t, sc) for _ in range(2)][1]       # (and every buffer is in torch's cache)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(4)]
    for s in streams:
        with torch.cuda.stream(s):
            torch.cuda._sleep(400_000_000)                           # one thread each, about 0.2 s
    got = bc.bitcos_pack_device(t, sc)
    running = [not s.query() for s in streams]
    torch.cuda.synchronize()
    assert all(running)
    assert torch.equal(got.signs, want.signs) and torch.equal(got.tile_off, want.tile_off) and torch.equal(got.bitmap, want.bitmap)


class CPack:
    """The C call with buffers of its own, so that a test sees all of them whatever the call returns."""

    def __init__(self, bc, t, sc, sign_bytes=None, stream=None):
        import ctypes as C
        self.bc, self.L, self.t, self.sc, (M, K) = bc, bc.load_library(), t, sc, t.shape
        n = [C.c_size_t(0) for _ in range(4)]
        assert self.L.bitcos_pack_sizes(M, K, int((t != 0).sum()), *[C.byref(v) for v in n]) == 0
        self.need = n[1].value
        self.sign_bytes = self.need if sign_bytes is None else sign_bytes(self.need)
        self.bitmap, self.off = (torch.full((v.value // 4,), -1, dtype=torch.int32, device="cuda") for v in (n[0], n[2]))
        self.signs = torch.full((self.sign_bytes // 4 + 16,), -1, dtype=torch.int32, device="cuda")
        self.scales = torch.full((n[3].value // 2,), -1, dtype=torch.int16, device="cuda")
        self.scratch = torch.empty(256, dtype=torch.uint8, device="cuda")
        self.off_host = torch.full((n[2].value // 4,), -1, dtype=torch.int32, pin_memory=True)
        self.stream = stream or torch.cuda.current_stream()
        torch.cuda.synchronize()

    def run(self, limit_ns=500_000_000):
        import ctypes as C
        nnz, launched, (M, K) = C.c_uint64(0), C.c_int(0), self.t.shape
        rc = self.L.bitcos_pack_device_limited(
            self.t.data_ptr(), self.sc.data_ptr(), M, K, self.bitmap.data_ptr(), self.signs.data_ptr(), self.sign_bytes, self.off.data_ptr(),
            self.scales.data_ptr(), self.off_host.data_ptr(), C.byref(nnz), self.scratch.data_ptr(), limit_ns, C.byref(launched),
            self.stream.cuda_stream)
        return rc, launched.value, nnz.value

    def equals(self, W):
        """All of this call's buffers against a packed matrix; nothing behind the sign vector was touched."""
        n, full = W.signs.numel(), self.sign_bytes // 16 * 4
        return (torch.equal(self.bitmap, W.bitmap) and torch.equal(self.off, W.tile_off) and torch.equal(self.scales, W.scales)
                and torch.equal(self.signs[:n], W.signs) and not self.signs[n:full].any() and bool((self.signs[full:] == -1).all())
                and np.array_equal(self.off_host.numpy()[:W.tile_off_host.size].view(np.uint32), W.tile_off_host))


def kernels(M, K):
    """How many kernels pack a matrix if no wait runs out."""
    return 1 if 6144 <= (M + 31) // 32 * (K // 128) <= 180224 else 3


def trits_and_scales(seed, M, K):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    t = torch.randint(-1, 2, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    return t, (0.01 + torch.rand((M, K // 128), generator=gen, device="cuda")).to(torch.bfloat16)


@pytest.mark.parametrize("M,K", [(300, 1280), (32 * 6143, 128), (32 * 6144, 128), (4097, 6144), (32 * 6513, 128), (25600, 5120)])
def test_device_pack_goes_on_when_its_wait_runs_out(bc, M, K):
    """With no time to wait every block but the first gives up; the call then packs in three kernels, and the same state serves the
    calls after it."""
    t, sc = trits_and_scales(31 + M + K, M, K)
    W = bc.bitcos_pack_device(t, sc)
    in_time = kernels(M, K)
    given_up = 4 if in_time == 1 else 3
    for limit, want in ((500_000_000, in_time), (0, given_up), (0, given_up), (500_000_000, in_time)):
        call = CPack(bc, t, sc)
        assert call.run(limit) == (0, want, W.nnz) and call.equals(W), limit
    bad = t.clone()
    bad[M - 1, K - 1] = 3
    assert CPack(bc, bad, sc).run(0)[:2] == (4, given_up)
    bad = sc.clone()
    bad[M - 1, 0] = -1.0
    assert CPack(bc, t, bad).run(0)[:2] == (5, given_up)
    assert CPack(bc, t, sc, lambda need: need - 16).run(0)[:2] == (6, given_up)


@pytest.mark.parametrize("M,K", [(96, 640), (2560, 2560), (8192, 5120)])
def test_device_pack_and_the_size_of_the_sign_vector(bc, M, K):
    """One bit short, exactly as large as needed, and larger: the error, and zeros up to the end of what was given."""
    t, sc = trits_and_scales(47 + M, M, K)
    W = bc.bitcos_pack_device(t, sc)
    for more, rc in ((-16, 6), (0, 0), (16, 0), (32 * 1024 + 48, 0), (2 * M * K // 8, 0)):
        call = CPack(bc, t, sc, lambda need: need + more)
        assert call.run()[:2] == (rc, kernels(M, K)), more
        if rc == 0:
            assert call.equals(W), more
        assert bool((call.signs[call.sign_bytes // 4:] == -1).all()), more


def test_device_pack_from_several_threads(bc):
    """Four host threads pack matrices of different sizes on streams of their own, over and over: every call has state of its own."""
    import threading
    jobs = [(trits_and_scales(61 + i, M, K), torch.cuda.Stream()) for i, (M, K) in enumerate(((8192, 5120), (2555, 6912), (25600, 5120), (96, 1280)))]
    want = [bc.bitcos_pack_device(t, sc) for (t, sc), _ in jobs]
    right = []

    def work(i):
        (t, sc), stream = jobs[i]
        with torch.cuda.stream(stream):
            for n in range(12):
                call = CPack(bc, t, sc, stream=stream)
                if call.run(0 if n % 4 == 3 else 500_000_000)[0] == 0 and call.equals(want[i]):
                    right.append((i, n))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert sorted(right) == [(i, n) for i in range(len(jobs)) for n in range(12)]


def test_device_pack_when_all_states_are_taken(bc):
    """Seventy calls at a time, held up behind a kernel that waits: 64 find a state, the others pack in three kernels."""
    import threading
    t, sc = trits_and_scales(71, 6144, 4096)
    want = bc.bitcos_pack_device(t, sc)
    n = 70
    calls = [CPack(bc, t, sc, stream=torch.cuda.Stream()) for _ in range(n)]
    ready, got = threading.Barrier(n + 1), [None] * n

    def work(i):
        ready.wait()
        got[i] = calls[i].run()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(n)]
    for th in threads:
        th.start()
    holder = torch.cuda.Stream()
    with torch.cuda.stream(holder):
        torch.cuda._sleep(1_500_000_000)                             # one thread, about 0.8 s
    for c in calls:
        if c.stream.cuda_stream != holder.cuda_stream:
            c.stream.wait_stream(holder)
    ready.wait()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert sorted(k for _, k, _ in got) == [1] * 64 + [3] * (n - 64)
    assert all(rc == 0 and nnz == want.nnz for rc, _, nnz in got) and all(c.equals(want) for c in calls)
