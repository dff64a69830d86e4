"""GPU parity: the CUDA library, called through its C ABI, against the CPU oracle.

Decompression must match the oracle bit for bit.  The fused calls accumulate in fp32 and are held
to |y - y_ref| <= 1e-3 * sum_i |w_i x_i| per output (y_ref = the oracle's fp64 sum over the
decompressed fp16 values); the plain relative error is also checked where |y_ref| is not small.
"""
import numpy as np
import pytest

from helpers import lib_meta_from_oracle, oracle_meta_from_lib, record_fused

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-3


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    from paper_2505_06901_b200 import binding

    binding.lib()
    return binding


@pytest.fixture(scope="module")
def W():
    from paper_2505_06901_b200 import workloads

    return workloads


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def gpu_decompress(B, lmeta, blocks):
    n = blocks.shape[0]
    d_meta = B.meta_to_device(lmeta)
    d_blocks = dev(blocks)
    d_out = torch.empty(max(n, 1) * 128, dtype=torch.float16, device="cuda")
    before = B.ecco_kernel_launch_count()
    B.ecco_decompress(d_meta, d_blocks, n, d_out)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    assert B.ecco_kernel_launch_count() == before + (1 if n else 0)
    return d_out[: n * 128].cpu().numpy().reshape(n, 128)


def assert_bit_exact(got, want):
    g, w = got.view(np.uint16), want.view(np.uint16)
    bad = np.nonzero((g != w).any(axis=1))[0]
    assert bad.size == 0, f"{bad.size} of {g.shape[0]} groups differ; first group {bad[:3]}, positions {np.nonzero(g[bad[0]] != w[bad[0]])[0][:8]}"


def gpu_gemv(B, lmeta, blocks, n_out, k, x, batch):
    d_meta, d_blocks, d_x = B.meta_to_device(lmeta), dev(blocks), dev(x)
    d_y = torch.full((batch, n_out), float("nan"), dtype=torch.float32, device="cuda")
    wsb = B.ecco_gemv_workspace_bytes(n_out, k, batch)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    ws.fill_(0xCD)                                   # stale contents must not matter
    B.ecco_gemv(d_meta, d_blocks, n_out, k, d_x, batch, d_y, ws, wsb)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    return d_y.cpu().numpy().astype(np.float64), (d_meta, d_blocks, d_x, ws, wsb)


def check_fused(got, ref, refabs, label="fused", tol=TOL, floor=1e-30):
    """|y - ref| <= tol sum|w x| + floor for every output, and the plain relative error <= 1e-3 wherever the reference is
    not small against its row (|ref| >= 0.1 rms); the largest values seen are kept for the session summary."""
    err = np.abs(got - ref)
    scaled = float((err / (refabs + floor / tol)).max())
    big = np.abs(ref) >= 0.1 * np.sqrt((ref ** 2).mean())
    plain = float((err[big] / np.abs(ref[big])).max()) if big.any() else 0.0
    record_fused(label, scaled, plain)
    assert np.all(err <= tol * refabs + floor), (label, scaled)
    assert plain <= TOL, (label, plain)


def test_calls_without_a_stream_go_to_the_current_one(B):
    """On the default stream, inside a stream context, after it and from another thread (whose current stream is its own)."""
    from concurrent.futures import ThreadPoolExecutor

    side = torch.cuda.Stream()
    assert B._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert B._stream(None) == side.cuda_stream
        with ThreadPoolExecutor(1) as ex:
            assert ex.submit(lambda: B._stream(None) == torch.cuda.current_stream().cuda_stream).result()
    assert B._stream(None) == torch.cuda.current_stream().cuda_stream


# ------------------------------------------------------------------ decompress
@pytest.mark.parametrize("e", [-32, -16, -15, 0, 7, 8, 16])
def test_decompress_every_scale_byte_at_the_edges_of_the_packed_product(B, eo, e):
    """The values of a group are packed fp16 products for 2^-15 <= T <= 2^7 and fp32 products outside: both sides of both
    edges, every scale byte (the two NaN codes among them), skewed codes so that all ranks, escapes and ends occur."""
    meta = make_meta(eo, skew_lens, e=e, seed=9)
    rb = np.random.Generator(np.random.PCG64(200 + e)).integers(0, 256, size=(1024, 64), dtype=np.uint8)
    rb[:, 0] = np.arange(1024) & 255
    got, want = gpu_decompress(B, lib_meta_from_oracle(B, meta), rb), eo.decode(meta, rb)
    assert_bit_exact(got, want)


@pytest.mark.parametrize("n_groups", [0, 1, 31, 32, 33, 1000, 1023, 1025, 2048])
def test_decompress_matches_oracle_ragged_sizes(B, eo, cfg1_small, n_groups):
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    blocks = cfg1_small["blocks"][:n_groups]
    got = gpu_decompress(B, lm, blocks)
    if n_groups:
        assert_bit_exact(got, eo.decode(cfg1_small["meta"], blocks))


def test_decompress_config1_full_with_library_metadata(B, eo, W):
    t = W.config1(keep_source=True)
    assert t.n_groups == 8192
    om = oracle_meta_from_lib(eo, t.meta)
    want_blocks, _ = eo.encode(om, t.source, eo.SELECT_MSE)
    assert np.array_equal(t.blocks, want_blocks)             # CPU encode: library == oracle
    got = gpu_decompress(B, t.meta, t.blocks)
    assert_bit_exact(got, eo.decode(om, t.blocks))
    src = t.source.astype(np.float32).reshape(-1, 128)
    rel = np.sqrt(((got.astype(np.float32) - src) ** 2).mean() / (src ** 2).mean())
    assert rel < 0.15


def test_decompress_kv_blocks_and_s16(B, eo, kv_small, synth):
    lm = lib_meta_from_oracle(B, kv_small["meta"])
    assert_bit_exact(gpu_decompress(B, lm, kv_small["blocks"]), eo.decode(kv_small["meta"], kv_small["blocks"]))
    # the paper's hardware compressor uses 16 patterns for the KV cache
    cal = synth.kv_cache(1, 4, 512, 2003, 3003)
    m16 = eo.calibrate(cal, S=16, H=4, seed=3, select=eo.SELECT_MINMAX)
    blocks, _ = eo.encode(m16, kv_small["k"], eo.SELECT_MINMAX)
    assert_bit_exact(gpu_decompress(B, lib_meta_from_oracle(B, m16), blocks), eo.decode(m16, blocks))


def test_decompress_is_total_on_garbage_and_edge_blocks(B, eo, cfg1_small, synth):
    meta = cfg1_small["meta"]
    lm = lib_meta_from_oracle(B, meta)
    rb = synth.random_blocks(4096, 99)
    assert_bit_exact(gpu_decompress(B, lm, rb), eo.decode(meta, rb))
    edge = np.stack([np.full(64, v, dtype=np.uint8) for v in (0x00, 0xFF, 0xAA, 0x55, 0x7F, 0x80)] * 8)
    assert_bit_exact(gpu_decompress(B, lm, edge), eo.decode(meta, edge))


def make_meta(eo, lens_fn, S=4, e=-5, seed=0):
    rng = np.random.Generator(np.random.PCG64(seed))
    m = eo.Meta()
    m.S, m.H, m.e = S, 4, e
    kl = eo.huffman_limited(np.ones(S), 12)
    for k in range(S):
        m.kp_len[k] = int(kl[k])
        pat = np.sort(rng.uniform(-1, 1, 15))
        for j in range(15):
            m.pattern[k][j] = int(np.float16(pat[j]).view(np.uint16))
        for h in range(4):
            ln = lens_fn(k, h, rng)
            for s in range(16):
                m.cb_len[k][h][s] = int(ln[s])
    assert eo.meta_check(m) == 0
    return m


def skew_lens(k, h, rng):
    """The most skewed admissible code (Kraft: 3/4 + 3/16 + 2/64 + 8/256 = 1).  Codebook 0 gives the
    2-bit codes to the middle centroids, where the values cluster (short streams, up to 16 pads); the
    other codebooks are random permutations (long streams, heavy clipping)."""
    lens = np.array([2, 2, 2, 4, 4, 4, 6, 6, 8, 8, 8, 8, 8, 8, 8, 8])
    out = np.zeros(16, dtype=np.int64)
    if h == 0:
        out[[7, 6, 8, 5, 9, 4, 10, 3, 11, 2, 12, 1, 13, 0, 14, 15]] = lens
    else:
        out[rng.permutation(16)] = lens
    return list(out)


def test_decompress_adversarial_codebooks(B, eo):
    """All-4-bit codes (10 + ID_KP + 128 x 4 > 512 bits: every group clips), the most skewed admissible
    code (2-bit symbols next to 8-bit ones: heavy clipping and up to 16 pads), long ID_KP codes,
    extreme exponents."""
    rng = np.random.Generator(np.random.PCG64(11))
    flat = make_meta(eo, lambda k, h, r: [4] * 16)
    skew = make_meta(eo, skew_lens, seed=3)
    for meta in (flat, skew):
        x = (rng.standard_t(3, size=(512, 128)) * 0.05).astype(np.float16)
        blocks, st = eo.encode(meta, x, eo.SELECT_MSE)
        got = gpu_decompress(B, lib_meta_from_oracle(B, meta), blocks)
        assert_bit_exact(got, eo.decode(meta, blocks))
        assert st.clipped_groups == st.n_groups if meta is flat else (st.padded_groups > 0 and st.clipped_groups > 0)
    # symbols forced to the longest codes -> every group clips; to the shortest -> 16 pads
    m = skew
    x = np.zeros((64, 128), dtype=np.float16)
    x[:, 0] = 1.0
    blocks, st = eo.encode(m, x, eo.SELECT_MSE)
    assert_bit_exact(gpu_decompress(B, lib_meta_from_oracle(B, m), blocks), eo.decode(m, blocks))
    for e in (-32, 16):
        m2 = make_meta(eo, lambda k, h, r: [4] * 16, e=e, seed=5)
        rb = np.random.Generator(np.random.PCG64(e + 100)).integers(0, 256, size=(256, 64), dtype=np.uint8)
        assert_bit_exact(gpu_decompress(B, lib_meta_from_oracle(B, m2), rb), eo.decode(m2, rb))
    # S = 64 with a deliberately unbalanced ID_KP code (lengths up to 12 bits)
    m3 = make_meta(eo, lambda k, h, r: [4] * 16, S=64, seed=7)
    kl = eo.huffman_limited(1.7 ** np.arange(64), 12)
    assert kl.max() == 12
    for k in range(64):
        m3.kp_len[k] = int(kl[k])
    assert eo.meta_check(m3) == 0
    rb = np.random.Generator(np.random.PCG64(8)).integers(0, 256, size=(2048, 64), dtype=np.uint8)
    assert_bit_exact(gpu_decompress(B, lib_meta_from_oracle(B, m3), rb), eo.decode(m3, rb))


def test_decompress_batch_matches_oracle_per_item(B, eo, cfg1_small, kv_small, synth):
    """One call over tensors with different metadata and sizes: every item as ecco_decompress alone would give it.
    Covers more than eight items (two launches), an empty item, tiny items (the small-tensor kernel in the middle
    of the batch) and a ragged tail; the items are independent of each other, as the call requires."""
    wm, km = cfg1_small["meta"], kv_small["meta"]
    d_wm, d_km = B.meta_to_device(lib_meta_from_oracle(B, wm)), B.meta_to_device(lib_meta_from_oracle(B, km))
    wb, kb = cfg1_small["blocks"], kv_small["blocks"]
    rb = synth.random_blocks(700, 5)
    plan = [(wm, d_wm, np.tile(wb, (3, 1))), (km, d_km, kb), (wm, d_wm, wb[:0]), (wm, d_wm, wb[:7]), (km, d_km, kb[:33]),
            (wm, d_wm, rb), (km, d_km, np.tile(kb, (2, 1))[:4095]), (wm, d_wm, wb[:1]), (km, d_km, kb[100:1124]),
            (wm, d_wm, wb[5:1030]), (km, d_km, kb[:31])]
    items, outs = [], []
    for meta, d_meta, blocks in plan:
        n = blocks.shape[0]
        d_b = dev(blocks) if n else torch.empty((1, 64), dtype=torch.uint8, device="cuda")
        d_o = torch.full((max(n, 1) * 128,), float("nan"), dtype=torch.float16, device="cuda")
        items.append((d_meta, d_b, n, d_o))
        outs.append(d_o)
    B.ecco_decompress_batch(items)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    for (meta, _, blocks), d_o in zip(plan, outs):
        n = blocks.shape[0]
        if n:
            assert_bit_exact(d_o[: n * 128].cpu().numpy().reshape(n, 128), eo.decode(meta, blocks))
    B.ecco_decompress_batch([])                                                   # nothing to do is not an error
    # one bad item stops the whole call before anything runs
    canary = torch.full((2048 * 128,), 7.0, dtype=torch.float16, device="cuda")
    with pytest.raises(B.EccoError) as ei:
        B.ecco_decompress_batch([(d_wm, dev(wb), 2048, canary), (d_wm, dev(wb).data_ptr() + 8, 2048, canary)])
    assert ei.value.code == B.ERR_ALIGNMENT
    torch.cuda.synchronize()
    assert bool((canary == 7.0).all())


@pytest.mark.parametrize("fill", ["ones", "random"])
@pytest.mark.parametrize("which", ["weights", "cache", "many shapes"])
def test_damaged_tables_give_unspecified_values_only(B, eo, cfg1_small, kv_small, synth, which, fill):
    """Any bytes in the tables that the decoders look up (ID_KP codes, shape and pair tables; the header and the records whole): lengths
    of up to 15 bits a symbol, so that lanes run on far behind their streams.  Every call still ends, writes its own output and nothing
    else, and the same call with the whole image is right afterwards.  The last warp's reads stay inside the CTA's shared memory: the
    static_assert at kFurthestRow."""
    from test_gpu_random import code_shapes

    all_shapes = code_shapes()                             # one to a codebook: an image without pair tables
    any_lens = lambda k, h, rng: list(rng.permutation(np.repeat(np.arange(2, 9), all_shapes[(4 * k + h) % len(all_shapes)])))
    meta = {"weights": cfg1_small["meta"], "cache": kv_small["meta"], "many shapes": make_meta(eo, any_lens, S=64, seed=6)}[which]
    whole = B.ecco_meta_serialize_device(lib_meta_from_oracle(B, meta))
    rng = np.random.Generator(np.random.PCG64(4))
    hdr = whole[:64].view(np.uint32)
    kp, rec, shape, pair = 64 + 64 * 32, 64 + 64 * 32 + 8192, 64 + 64 * 32 + 8192 + 4096 + 8320, int(hdr[11])     # csrc/ecco_format.h
    assert pair >= shape + int(hdr[8]) and pair + int(hdr[9]) == whole.size and (hdr[9] == 0) == (which == "many shapes")
    damaged = whole.copy()
    for lo, hi in ((kp, rec), (shape, shape + int(hdr[8])), (pair, whole.size)):
        damaged[lo:hi] = 0xFF if fill == "ones" else rng.integers(0, 256, hi - lo, dtype=np.uint8)
    n_out, k, heads, seq, qpk = 256, 1024, 4, 512, 8
    blocks, n = synth.random_blocks(2048, 11), 2048
    lm = lib_meta_from_oracle(B, meta)
    x16 = synth.weight_matrix(256, 1024, 1001)
    stream, index, _ = B.ecco_var_encode_host(lm, x16, B.SELECT_MSE | B.KEEP_EXPONENT)
    d_blocks, d_stream, d_index = dev(blocks), dev(stream), dev(index)
    d_x, d_q, d_s = dev(synth.activations(8, k, 3)), dev(synth.queries(1, heads * qpk, 4)), torch.zeros((1, heads * qpk, seq), device="cuda")
    ws = torch.empty(max(B.ecco_gemv_workspace_bytes(n_out, k, 8), B.ecco_attn_values_workspace_bytes(1, heads, seq, qpk)), dtype=torch.uint8, device="cuda")

    def calls(image):
        d_meta, outs = dev(image), []

        def out(count, dtype):                             # with a margin that nobody may write
            t = torch.full((count + 4096,), 7.0, dtype=dtype, device="cuda")
            outs.append((t, count))
            return t
        B.ecco_decompress(d_meta, d_blocks, n, out(n * 128, torch.float16))
        B.ecco_decompress(d_meta, d_blocks, 31, out(31 * 128, torch.float16))
        B.ecco_var_decompress(d_meta, d_stream, d_index, n, out(n * 128, torch.float16))
        for batch in (1, 4, 8):
            B.ecco_gemv(d_meta, d_blocks, n_out, k, d_x, batch, out(batch * n_out, torch.float32), ws, ws.numel())
        for q in (1, 8):
            B.ecco_attn_scores(d_meta, d_blocks, 1, heads, seq, q, d_q, 0.5, out(heads * q * seq, torch.float32))
            B.ecco_attn_values(d_meta, d_blocks, 1, heads, seq, q, d_s, out(heads * q * 128, torch.float32), ws, ws.numel())
        assert B.ecco_device_status() == 0
        assert all(bool((t[c:] == 7.0).all()) for t, c in outs)
        return outs

    want = calls(whole)
    assert_bit_exact(want[0][0][: n * 128].cpu().numpy().reshape(n, 128), eo.decode(meta, blocks))
    calls(damaged)
    assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for (a, _), (b, _) in zip(calls(whole), want))


@pytest.mark.parametrize("n_groups", [32, 33, 700])
def test_decompress_batch_of_short_tensors_with_tables_of_their_own(B, eo, cfg1_small, kv_small, synth, n_groups):
    """Eight runs in one launch, each with other tables than the one before and its arrays elsewhere: most warps
    help with the tables of a run and have no tile in it.  Repeated, in two orders; exact: decoding has one result."""
    shapes = np.array([[2, 2, 2, 4, 4, 4, 6, 6, 8, 8, 8, 8, 8, 8, 8, 8], [4] * 16])
    metas = [cfg1_small["meta"], kv_small["meta"], make_meta(eo, skew_lens, S=7, seed=4), make_meta(eo, lambda k, h, r: list(r.permutation(shapes[k & 1])), S=64, seed=6)]
    plan = []
    for i in range(8):
        m = metas[i % 4].copy()
        blocks = synth.random_blocks(n_groups, 60 + i)
        plan.append((B.meta_to_device(lib_meta_from_oracle(B, m)), dev(blocks), dev(eo.decode(m, blocks))))
    outs = [torch.empty((n_groups, 128), dtype=torch.float16, device="cuda") for _ in plan]
    for order in (range(8), (3, 0, 2, 1, 7, 6, 5, 4)):
        items = B.decompress_items([(plan[i][0], plan[i][1], n_groups, outs[i]) for i in order])
        for _ in range(20):
            for o in outs:
                o.fill_(7.0)
            B.ecco_decompress_batch(items)
            assert all(torch.equal(o.view(torch.int16), p[2].view(torch.int16)) for o, p in zip(outs, plan))
    assert B.ecco_device_status() == 0


def test_decompress_every_code_shape_on_random_streams(B, eo, synth):
    """All 255 admissible shapes of a 2..8-bit code on 16 symbols (every multiset of lengths with Kraft sum 1,
    dealt to the symbols at random), one per codebook, decoded from random bit streams: whatever a block's header
    bits select, table lookups and arithmetic decoding must give the oracle's values, clips and outliers."""
    shapes = []

    def rec(L, left, kraft, counts):
        if L == 9:
            if left == 0 and kraft == 0:
                shapes.append(tuple(counts))
            return
        worth = 1 << (8 - L)
        for c in range(min(left, kraft // worth) + 1):
            rec(L + 1, left - c, kraft - c * worth, counts + [c])

    rec(2, 16, 256, [])
    assert len(shapes) == 255
    rng = np.random.Generator(np.random.PCG64(99))
    m = eo.Meta()
    m.S, m.H, m.e = 64, 4, -3
    kl = eo.huffman_limited(np.ones(64), 12)
    for k in range(64):
        m.kp_len[k] = int(kl[k])
        pat = np.sort(rng.uniform(-1, 1, 15))
        for j in range(15):
            m.pattern[k][j] = int(np.float16(pat[j]).view(np.uint16))
        for h in range(4):
            lens = rng.permutation(np.repeat(np.arange(2, 9), shapes[(k * 4 + h) % len(shapes)]))
            for s in range(16):
                m.cb_len[k][h][s] = int(lens[s])
    assert eo.meta_check(m) == 0
    rb = synth.random_blocks(32 * 1024, 31)
    lm = lib_meta_from_oracle(B, m)
    assert_bit_exact(gpu_decompress(B, lm, rb), eo.decode_threads(m, rb, 8))
    # the fused consumers over the same streams (their decoder is all-table; one and eight rows of x take the
    # scalar and the tensor-core kernel)
    for batch in (1, 8):
        x = synth.activations(batch, 2048, 40 + batch)
        got, _ = gpu_gemv(B, lm, rb, 2048, 2048, x, batch)
        ref, refabs = eo.gemv(m, rb, 2048, 2048, x, batch)
        check_fused(got, ref, refabs, f"gemv b{batch} code shapes")


def test_decompress_rejects_bad_arguments_on_device(B, cfg1_small):
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    d_meta, d_blocks = B.meta_to_device(lm), dev(cfg1_small["blocks"])
    d_out = torch.empty(2048 * 128 + 8, dtype=torch.float16, device="cuda")
    L = B.lib()
    assert L.ecco_decompress(d_meta.data_ptr(), d_blocks.data_ptr(), 10, d_out.data_ptr() + 2, None) == B.ERR_ALIGNMENT
    assert L.ecco_decompress(d_meta.data_ptr(), d_blocks.data_ptr() + 8, 10, d_out.data_ptr(), None) == B.ERR_ALIGNMENT
    assert L.ecco_decompress(None, d_blocks.data_ptr(), 10, d_out.data_ptr(), None) == B.ERR_INVALID_ARG
    # a side stream works like the current one
    s = torch.cuda.Stream()
    B.ecco_decompress(d_meta, d_blocks, 2048, d_out, stream=s)
    s.synchronize()
    assert B.ecco_device_status() == 0


def test_bounded_wait_gives_up_and_reports(B, eo, cfg1_small):
    """The device-side wait on the table copy is bounded: when it runs out the kernel records
    ECCO_ERR_DEVICE_TIMEOUT and returns, ecco_device_status reports it once, and the context stays usable."""
    assert B.ecco_device_status() == 0
    B.ecco_test_wait_timeout()
    assert B.ecco_device_status() == B.ERR_DEVICE_TIMEOUT
    assert B.ecco_device_status() == 0                      # reading clears it
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    assert_bit_exact(gpu_decompress(B, lm, cfg1_small["blocks"][:100]), eo.decode(cfg1_small["meta"], cfg1_small["blocks"][:100]))


# ------------------------------------------------------------------ fused GEMV
@pytest.mark.parametrize("n_out,k,batch", [(256, 1024, 1), (256, 1024, 3), (256, 1024, 8), (100, 1024, 2), (513, 512, 5),
                                           (2048, 128, 1), (64, 4096, 4), (1, 128, 1)])
def test_gemv_matches_oracle(B, eo, cfg1_small, synth, n_out, k, batch):
    meta = cfg1_small["meta"]
    n_groups = n_out * (k // 128)
    reps = -(-n_groups // 2048)
    blocks = np.tile(cfg1_small["blocks"], (reps, 1))[:n_groups]
    x = synth.activations(batch, k, 50 + n_out + batch)
    got, keep = gpu_gemv(B, lib_meta_from_oracle(B, meta), blocks, n_out, k, x, batch)
    ref, refabs = eo.gemv(meta, blocks, n_out, k, x, batch)
    check_fused(got, ref, refabs, f"gemv b{batch}")
    # a second call on the same (now dirty) workspace gives the same bits: fixed summation order
    d_meta, d_blocks, d_x, ws, wsb = keep
    d_y2 = torch.empty((batch, n_out), dtype=torch.float32, device="cuda")
    B.ecco_gemv(d_meta, d_blocks, n_out, k, d_x, batch, d_y2, ws, wsb)
    torch.cuda.synchronize()
    assert np.array_equal(d_y2.cpu().numpy().astype(np.float64), got)


def test_gemv_handles_pads_clips_and_garbage(B, eo, cfg1_small, synth):
    meta = cfg1_small["meta"]
    rb = synth.random_blocks(512 * 4, 123)                 # garbage streams: duplicate pad locations etc.
    x = synth.activations(8, 512, 9)
    got, _ = gpu_gemv(B, lib_meta_from_oracle(B, meta), rb, 512, 512, x, 8)
    ref, refabs = eo.gemv(meta, rb, 512, 512, x, 8)
    check_fused(got, ref, refabs, "gemv b8 garbage")
    skew = make_meta(eo, skew_lens, seed=3)   # many pads, many clips
    w = (np.random.Generator(np.random.PCG64(1)).standard_t(3, size=(256, 256)) * 0.05).astype(np.float16)
    blocks, st = eo.encode(skew, w, eo.SELECT_MSE)
    assert st.padded_values > st.n_groups and st.clipped_groups > 0
    x = synth.activations(2, 256, 10)
    got, _ = gpu_gemv(B, lib_meta_from_oracle(B, skew), blocks, 256, 256, x, 2)
    ref, refabs = eo.gemv(skew, blocks, 256, 256, x, 2)
    check_fused(got, ref, refabs, "gemv b2 skewed code")


@pytest.mark.parametrize("batch", [3, 4, 5, 6])
@pytest.mark.parametrize("n_out,k", [(33, 2048), (2047, 512), (4999, 640)])
def test_gemv_of_three_to_six_rows(B, eo, cfg1_small, synth, batch, n_out, k):
    """Either side of the line between the per-warp and the tensor-core kernel: one tile of rows split between many warps, and
    calls with more units than warps, with a ragged last tile."""
    meta = cfg1_small["meta"]
    n = n_out * k // 128
    blocks = np.tile(cfg1_small["blocks"], (-(-n // len(cfg1_small["blocks"])), 1))[:n]
    x = synth.activations(batch, k, 90 + batch)
    got, _ = gpu_gemv(B, lib_meta_from_oracle(B, meta), blocks, n_out, k, x, batch)
    ref, refabs = eo.gemv(meta, blocks, n_out, k, x, batch)
    check_fused(got, ref, refabs, f"gemv b{batch}")


@pytest.mark.parametrize("batch", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n_out,k", [(513, 512), (999, 4096)])
def test_gemv_error_does_not_grow_with_the_rows_of_x(B, eo, cfg1_small, synth, batch, n_out, k):
    """Calls of one k-block per warp, 2-norm of the error over that of the result.  An addition is off by 0.43 * 2^-24 of its result
    (rms: half a last place is 2^-25..2^-24 of a number, its uniform error 1 / sqrt(3) of that), so a chain of n products of random
    sign by that times sqrt(n / 2).  Two chains of 64 make a k-block's 128 products and one of k / 128 the partial sums; the limit lies
    halfway to a single chain of 128, i.e. at 96."""
    n = n_out * (k // 128)
    blocks = np.tile(cfg1_small["blocks"], (-(-n // 2048), 1))[:n]
    x = synth.activations(batch, k, 7)
    got, _ = gpu_gemv(B, lib_meta_from_oracle(B, cfg1_small["meta"]), blocks, n_out, k, x, batch)
    ref, _ = eo.gemv(cfg1_small["meta"], blocks, n_out, k, x, batch)
    rel = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    assert rel <= 0.43 * 2.0 ** -24 * np.sqrt((96 + k // 128) / 2), rel


@pytest.mark.parametrize("batch", [1, 3, 5, 8])
def test_gemv_numbers_that_are_not_finite_stay_in_their_sums(B, eo, cfg1_small, synth, batch):
    """An infinity or a NaN in one row of x, under mapped values and under outliers: that row's outputs are not finite, the others are
    what they are without it, bit for bit."""
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    n_out, k = 256, 1024
    x = synth.activations(batch, k, 9)
    clean, _ = gpu_gemv(B, lm, cfg1_small["blocks"], n_out, k, x, batch)
    for bad in (np.inf, -np.inf, np.nan):
        for at in (0, 517, 1023):
            y = x.copy()
            y[batch // 2, at] = bad
            got, _ = gpu_gemv(B, lm, cfg1_small["blocks"], n_out, k, y, batch)
            assert not np.isfinite(got[batch // 2]).any()
            rest = np.arange(batch) != batch // 2
            assert np.array_equal(got[rest], clean[rest])


@pytest.mark.parametrize("batch", [1, 2, 3, 8])
def test_gemv_batch_gives_every_item_what_gemv_gives(B, eo, cfg1_small, synth, batch):
    """Several matrices in one call (shapes that differ in rows and in k, a ragged row count, a one-row matrix, a shared
    x, per-tensor exponents that differ): every item within the fused tolerance of the oracle and, to rounding, what
    ecco_gemv gives on it alone (the k range of a row is cut into partial sums at other places, so the last bits may
    differ); the same call twice gives the same bits.  Eight items is the most one call takes."""
    meta = cfg1_small["meta"]
    shapes = [(256, 1024), (100, 1024), (513, 512), (64, 4096), (1, 128), (2048, 128), (31, 256), (96, 1024)]
    x_shared = synth.activations(batch, 1024, 77)
    items, keep, want = [], [], []
    for i, (n_out, k) in enumerate(shapes):
        n_groups = n_out * (k // 128)
        blocks = np.roll(np.tile(cfg1_small["blocks"], (-(-n_groups // 2048), 1)), 17 * i, axis=0)[:n_groups]
        om = meta.copy()
        om.e = meta.e + (i % 3) - 1                           # same tables, another exponent
        x = x_shared if k == 1024 else synth.activations(batch, k, 80 + i)
        d_meta, d_blocks, d_x = B.meta_to_device(lib_meta_from_oracle(B, om)), dev(blocks), dev(x)
        d_y = torch.full((batch, n_out), float("nan"), dtype=torch.float32, device="cuda")
        items.append((d_meta, d_blocks, n_out, k, d_x, d_y))
        keep.append((om, blocks, x))
        wsb = B.ecco_gemv_workspace_bytes(n_out, k, batch)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        d_alone = torch.empty((batch, n_out), dtype=torch.float32, device="cuda")
        B.ecco_gemv(d_meta, d_blocks, n_out, k, d_x, batch, d_alone, ws, wsb)
        want.append(d_alone)
    wsb = B.ecco_gemv_batch_workspace_bytes(items, batch)
    assert wsb > 0
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    first = None
    for _ in range(2):                                        # the second call starts from a used workspace
        B.ecco_gemv_batch(items, batch, ws, wsb)
        torch.cuda.synchronize()
        assert B.ecco_device_status() == 0
        outs = [it[5].cpu().numpy() for it in items]
        if first is not None:
            assert all(np.array_equal(a, b) for a, b in zip(first, outs))
        first = outs
    for (om, blocks, x), it, alone, got in zip(keep, items, want, first):
        ref, refabs = eo.gemv(om, blocks, it[2], it[3], x, batch)
        check_fused(got.astype(np.float64), ref, refabs, f"gemv batch-call b{batch}")
        assert np.all(np.abs(got - alone.cpu().numpy()) <= 1e-5 * refabs + 1e-30)
    # argument errors stop the call before anything runs; too small a workspace is refused
    with pytest.raises(B.EccoError) as ei:
        B.ecco_gemv_batch(items + items[:1], batch, ws, wsb)
    assert ei.value.code == B.ERR_INVALID_ARG
    with pytest.raises(B.EccoError) as ei:
        B.ecco_gemv_batch(items, batch, ws, wsb - 256)
    assert ei.value.code == B.ERR_WORKSPACE
    # an item with other decode tables is detected on the device: nothing is written, the status says so
    S, e, pat, cb, kp = lib_meta_from_oracle(B, meta).tables()
    cb = cb.copy()
    cb[0, 0] = cb[0, 0][::-1]
    other = B.meta_to_device(B.ecco_meta_create(S, e, pat, cb, kp))
    canary = torch.full((batch, shapes[0][0]), 7.0, dtype=torch.float32, device="cuda")
    bad = [(items[0][0], items[0][1], items[0][2], items[0][3], items[0][4], canary),
           (other, items[1][1], items[1][2], items[1][3], items[1][4], items[1][5])]
    B.ecco_gemv_batch(bad, batch, ws, wsb)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == B.ERR_INVALID_ARG
    assert B.ecco_device_status() == 0                        # reported once
    assert bool((canary == 7.0).all())
    B.ecco_gemv_batch(items, batch, ws, wsb)                  # and the next good call is unaffected
    torch.cuda.synchronize()
    assert np.array_equal(items[0][5].cpu().numpy(), first[0])


def test_gemv_workspace_errors(B, cfg1_small, synth):
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    d_meta, d_blocks = B.meta_to_device(lm), dev(cfg1_small["blocks"])
    d_x, d_y = dev(synth.activations(1, 1024, 1)), torch.empty((1, 256), dtype=torch.float32, device="cuda")
    with pytest.raises(B.EccoError) as ei:
        B.ecco_gemv(d_meta, d_blocks, 256, 1024, d_x, 1, d_y, None, 0)
    assert ei.value.code == B.ERR_WORKSPACE
    small = torch.empty(64, dtype=torch.uint8, device="cuda")
    with pytest.raises(B.EccoError) as ei:
        B.ecco_gemv(d_meta, d_blocks, 256, 1024, d_x, 1, d_y, small, 64)
    assert ei.value.code == B.ERR_WORKSPACE


@pytest.mark.parametrize("n_out,k,batch", [(32, 128, 1), (40, 8192, 1), (4096, 1024, 2), (96, 16384, 3), (513, 4096, 8)])
def test_gemv_does_not_care_what_the_workspace_holds(B, eo, cfg1_small, synth, n_out, k, batch):
    """Row tiles of one warp, of a few and of a hundred: the same bits from a workspace of zeros, of ones, of random words and of
    what earlier calls left in it (an odd number of calls later, and after a call of another shape)."""
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    n = n_out * (k // 128)
    blocks = np.tile(cfg1_small["blocks"], (-(-n // 2048), 1))[:n]
    d_meta, d_blocks, d_x = B.meta_to_device(lm), dev(blocks), dev(synth.activations(batch, k, 5))
    wsb = max(B.ecco_gemv_workspace_bytes(n_out, k, batch), B.ecco_gemv_workspace_bytes(64, 256, batch))
    first = None
    for fill in (0, 0xFF, None, "left", "left", "other"):
        if fill == "other":
            B.ecco_gemv(d_meta, d_blocks, 32, 128, d_x, batch, torch.empty((batch, 32), device="cuda"), ws, wsb)
        elif fill != "left":
            ws = torch.randint(0, 256, (wsb,), dtype=torch.uint8, device="cuda") if fill is None else torch.full((wsb,), fill, dtype=torch.uint8, device="cuda")
        y = torch.full((batch, n_out), float("nan"), dtype=torch.float32, device="cuda")
        B.ecco_gemv(d_meta, d_blocks, n_out, k, d_x, batch, y, ws, wsb)
        first = y if first is None else first
        assert torch.equal(y, first), fill
    ref, refabs = eo.gemv(cfg1_small["meta"], blocks[: n], n_out, k, synth.activations(batch, k, 5), batch)
    check_fused(first.cpu().numpy().astype(np.float64), ref, refabs, f"gemv b{batch} workspaces")


def counts_left(ws, partial_floats, stride, n):
    """The counts in the ticket words of a workspace: the low 16 bits of n 64-bit words, `stride` words apart, behind the partial sums."""
    at = -(-partial_floats * 4 // 256) * 256
    return ws[at: at + 8 * stride * n].cpu().numpy().view(np.uint64)[::stride] & np.uint64(0xFFFF)


@pytest.mark.parametrize("batch", [1, 8])
@pytest.mark.parametrize("n_out,k", [(40, 4096), (96, 640), (32, 8192)])
def test_gemv_blocks_that_give_up_leave_no_count(B, cfg1_small, synth, batch, n_out, k):
    """A CTA whose table fetch times out passes the tickets of the row tiles it shares: a word left with a count would be wrong at
    every replay of a captured call.  At most 64 units, so every unit has a CTA and a slot of its own."""
    n = n_out * (k // 128)
    tiles = -(-n_out // 32)
    units = tiles * (k // 128)
    blocks = np.tile(cfg1_small["blocks"], (-(-n // 2048), 1))[:n]
    y = torch.empty((batch, n_out), device="cuda")
    items = [(B.meta_to_device(lib_meta_from_oracle(B, cfg1_small["meta"])), dev(blocks), n_out, k, dev(synth.activations(batch, k, 3)), y)]
    wsb = B.ecco_gemv_batch_workspace_bytes(items, batch)
    ws = torch.zeros(wsb, dtype=torch.uint8, device="cuda")
    B.ecco_gemv_batch(items, batch, ws, wsb)
    want = y.clone()
    for _ in range(3):
        B.ecco_test_gemv_give_up(items, batch, ws, wsb)
        torch.cuda.synchronize()
        assert B.ecco_device_status() == B.ERR_DEVICE_TIMEOUT
        words = ws.view(torch.int64)
        assert bool((words != 0).any())
        assert not counts_left(ws, (units + tiles) * (1 if batch == 1 else 8) * 32, 4, tiles).any()
        B.ecco_gemv_batch(items, batch, ws, wsb)
        assert torch.equal(y, want) and B.ecco_device_status() == 0


def test_attn_values_blocks_that_give_up_leave_no_count(B, kv_small):
    """The same for the heads that CTAs share: two rows of 20 tiles, one tile to a CTA."""
    heads, seq, qpk = 2, 640, 4
    blocks = kv_small["blocks"][: heads * seq]
    scores = np.random.Generator(np.random.PCG64(1)).standard_normal((1, heads * qpk, seq)).astype(np.float32)
    out = torch.empty((1, heads * qpk, 128), device="cuda")
    wsb = B.ecco_attn_values_workspace_bytes(1, heads, seq, qpk)
    ws = torch.zeros(wsb, dtype=torch.uint8, device="cuda")
    args = (B.meta_to_device(lib_meta_from_oracle(B, kv_small["meta"])), dev(blocks), 1, heads, seq, qpk, dev(scores), out, ws, wsb)
    B.ecco_attn_values(*args)
    want = out.clone()
    for _ in range(3):
        B.ecco_test_attn_values_give_up(*args)
        torch.cuda.synchronize()
        assert B.ecco_device_status() == B.ERR_DEVICE_TIMEOUT
        assert not counts_left(ws, (heads * 20 + heads) * (128 * 8 + 16), 1, heads).any()
        B.ecco_attn_values(*args)
        assert torch.equal(out, want) and B.ecco_device_status() == 0


# ------------------------------------------------------------------ fused attention scores
@pytest.mark.parametrize("batch,heads,seq,qpk", [(2, 4, 256, 1), (2, 4, 256, 2), (2, 4, 256, 8), (1, 3, 77, 4), (1, 1, 1, 1),
                                                 (2, 2, 513, 3)])
def test_attn_scores_match_oracle(B, eo, kv_small, synth, batch, heads, seq, qpk):
    meta = kv_small["meta"]
    n = batch * heads * seq
    blocks = np.tile(kv_small["blocks"], (-(-n // 2048), 1))[:n]
    q = synth.queries(batch, heads * qpk, 60 + seq)
    scale = 128 ** -0.5
    d_meta, d_blocks, d_q = B.meta_to_device(lib_meta_from_oracle(B, meta)), dev(blocks), dev(q)
    d_s = torch.full((batch, heads * qpk, seq), float("nan"), dtype=torch.float32, device="cuda")
    B.ecco_attn_scores(d_meta, d_blocks, batch, heads, seq, qpk, d_q, scale, d_s)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    ref, refabs = eo.attn_scores(meta, blocks, batch, heads, seq, qpk, q, scale)
    check_fused(d_s.cpu().numpy().astype(np.float64), ref, refabs, f"scores q{qpk}")


@pytest.mark.parametrize("seq", [1, 31, 32, 33, 200])
def test_many_outliers_and_repeated_locations(B, eo, synth, seq):
    """Groups of short codewords with random bits where the outlier fields sit: up to 480 outliers per warp (several rounds of
    dealing them out), locations that occur twice (the later field wins), next to groups with few outliers and with none."""
    rng = np.random.Generator(np.random.PCG64(900 + seq))
    meta = make_meta(eo, skew_lens, seed=3)
    heads, n = 3, 3 * seq
    x = (rng.standard_normal((n, 128)) * 0.01).astype(np.float16)
    x[:, 0] = 1.0                                          # everything else near zero: two-bit codewords
    few = rng.random(n) < 0.3
    x[few] = (rng.standard_t(3, size=(int(few.sum()), 128)) * 0.05).astype(np.float16)
    blocks, st = eo.encode(meta, x, eo.SELECT_MSE)
    _, _, info = eo.decode_block(meta, blocks[int(np.argmin(few))])
    assert st.padded_groups > 0 and (few.all() or info.n_pad >= 15)
    many = np.array([eo.decode_block(meta, b)[2].n_pad >= 15 for b in blocks])
    blocks[np.ix_(many, range(36, 64))] = rng.integers(0, 256, size=(int(many.sum()), 28), dtype=np.uint8)
    lm = lib_meta_from_oracle(B, meta)
    assert_bit_exact(gpu_decompress(B, lm, blocks), eo.decode(meta, blocks))
    d_meta, d_blocks = B.meta_to_device(lm), dev(blocks)
    for qpk in (1, 2, 3, 8):
        q = synth.queries(1, heads * qpk, 60 + qpk)
        d_s = torch.full((1, heads * qpk, seq), float("nan"), dtype=torch.float32, device="cuda")
        B.ecco_attn_scores(d_meta, d_blocks, 1, heads, seq, qpk, dev(q), 0.5, d_s)
        torch.cuda.synchronize()
        ref, refabs = eo.attn_scores(meta, blocks, 1, heads, seq, qpk, q, 0.5)
        check_fused(d_s.cpu().numpy().astype(np.float64), ref, refabs, f"scores q{qpk} outliers")
    for batch in (1, 2, 3):
        a = synth.activations(batch, 128, seq)
        got, _ = gpu_gemv(B, lm, blocks, n, 128, a, batch)
        ref, refabs = eo.gemv(meta, blocks, n, 128, a, batch)
        check_fused(got, ref, refabs, f"gemv b{batch} outliers")


# ------------------------------------------------------------------ full-size configurations
def host_threads():
    import os

    return max(1, len(os.sched_getaffinity(0)))


def sample_groups(n, rng, k=6144):
    idx = np.unique(np.concatenate([np.arange(min(n, 1024)), np.arange(max(0, n - 1024), n), rng.integers(0, n, k)]))
    return idx


def assert_device_equals_oracle(eo, om, blocks, d_out):
    """Every group of the tensor: the oracle decodes all of them on the host cores, the comparison runs on the GPU."""
    n = blocks.shape[0]
    want = eo.decode_threads(om, blocks, host_threads()).view(np.int16)
    d_want = torch.from_numpy(want).cuda()
    got = d_out.view(torch.int16).view(n, 128)
    if not torch.equal(got, d_want):
        bad = torch.nonzero((got != d_want).any(dim=1)).flatten()
        g = int(bad[0])
        raise AssertionError(f"{bad.numel()} of {n} groups differ; first group {g}, positions "
                             f"{torch.nonzero(got[g] != d_want[g]).flatten()[:8].tolist()}")


def check_full_decompress(B, eo, t, d_out=None):
    d_meta, d_blocks = B.meta_to_device(t.meta), dev(t.blocks)
    d_out = torch.empty(t.n_groups * 128, dtype=torch.float16, device="cuda")
    B.ecco_decompress(d_meta, d_blocks, t.n_groups, d_out)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    om = oracle_meta_from_lib(eo, t.meta)
    assert_device_equals_oracle(eo, om, t.blocks, d_out)
    return om, d_meta, d_blocks


def oracle_gemv_threads(eo, om, blocks, n_out, k, x, batch):
    """eo.gemv over disjoint row ranges from one Python thread per host core (ctypes drops the GIL)."""
    from concurrent.futures import ThreadPoolExecutor

    kb = k // 128
    threads = min(host_threads(), n_out)
    bounds = [n_out * i // threads for i in range(threads + 1)]
    ref, refabs = np.zeros((batch, n_out)), np.zeros((batch, n_out))

    def work(i):
        lo, hi = bounds[i], bounds[i + 1]
        if hi > lo:
            r, a = eo.gemv(om, blocks[lo * kb:hi * kb], hi - lo, k, x, batch)
            ref[:, lo:hi], refabs[:, lo:hi] = r, a

    with ThreadPoolExecutor(threads) as ex:
        list(ex.map(work, range(threads)))
    return ref, refabs


def check_full_gemv(B, eo, synth, t, om, d_meta, d_blocks, batch, all_rows=False):
    n_out, k = t.shape
    x = synth.activations(batch, k, 70 + batch)
    d_x = dev(x)
    d_y = torch.empty((batch, n_out), dtype=torch.float32, device="cuda")
    wsb = B.ecco_gemv_workspace_bytes(n_out, k, batch)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    B.ecco_gemv(d_meta, d_blocks, n_out, k, d_x, batch, d_y, ws, wsb)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    y = d_y.cpu().numpy().astype(np.float64)
    if all_rows:
        ref, refabs = oracle_gemv_threads(eo, om, t.blocks, n_out, k, x, batch)
        check_fused(y, ref, refabs, f"gemv b{batch} full {n_out}x{k}")
        return
    rows = np.unique(np.concatenate([[0, n_out - 1], np.random.Generator(np.random.PCG64(n_out + batch)).integers(0, n_out, 48)]))
    kb = k // 128
    sub = np.concatenate([t.blocks[r * kb:(r + 1) * kb] for r in rows])
    ref, refabs = eo.gemv(om, sub, len(rows), k, x, batch)
    check_fused(y[:, rows], ref, refabs, f"gemv b{batch} full {n_out}x{k}")


def test_config2_llama7b_layer_full_size(B, eo, W, synth):
    items, metas = [], []
    for t in W.config2(names=("q", "gate", "down")):
        om, d_meta, d_blocks = check_full_decompress(B, eo, t)
        for batch in (1, 8):                               # every output row against the oracle's fp64 product
            check_full_gemv(B, eo, synth, t, om, d_meta, d_blocks, batch, all_rows=True)
        items.append((d_meta, d_blocks, t.n_groups, torch.empty(t.n_groups * 128, dtype=torch.float16, device="cuda")))
        metas.append((om, t))
    # the three tensors in the launch configuration bench.py times: one batched call (one run: the tensors share
    # their tables and differ in the exponent), every group against the oracle
    B.ecco_decompress_batch(items)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    for (om, t), (_, _, n, d_out) in zip(metas, items):
        assert_device_equals_oracle(eo, om, t.blocks, d_out)
    # the fused GEMV in the launch configuration bench.py times: matrices that share x in one ecco_gemv_batch call
    # (here q with itself standing in for k and v, and gate twice for gate + up), every output row against the oracle
    (oq, tq), (og, tg) = metas[0], metas[1]
    for batch in (1, 8):
        for om, t, (d_meta, d_blocks, _, _), copies in ((oq, tq, items[0], 3), (og, tg, items[1], 2)):
            n_out, k = t.shape
            x = synth.activations(batch, k, 90 + batch)
            d_x = dev(x)
            ys = [torch.full((batch, n_out), float("nan"), dtype=torch.float32, device="cuda") for _ in range(copies)]
            call = [(d_meta, d_blocks, n_out, k, d_x, y) for y in ys]
            wsb = B.ecco_gemv_batch_workspace_bytes(call, batch)
            ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
            B.ecco_gemv_batch(call, batch, ws, wsb)
            torch.cuda.synchronize()
            assert B.ecco_device_status() == 0
            ref, refabs = oracle_gemv_threads(eo, om, t.blocks, n_out, k, x, batch)
            for y in ys:
                check_fused(y.cpu().numpy().astype(np.float64), ref, refabs, f"gemv batch-call b{batch} full {n_out}x{k}")


def check_full_attn(B, eo, synth, t, qpk):
    batch, heads, seq, _ = t.shape
    om = oracle_meta_from_lib(eo, t.meta)
    q = synth.queries(batch, heads * qpk, 80 + qpk)
    d_meta, d_blocks, d_q = B.meta_to_device(t.meta), dev(t.blocks), dev(q)
    d_s = torch.empty((batch, heads * qpk, seq), dtype=torch.float32, device="cuda")
    B.ecco_attn_scores(d_meta, d_blocks, batch, heads, seq, qpk, d_q, 128 ** -0.5, d_s)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    s = d_s.cpu().numpy().astype(np.float64)
    rng = np.random.Generator(np.random.PCG64(seq + qpk))
    for _ in range(6):
        b, h = int(rng.integers(batch)), int(rng.integers(heads))
        t0 = int(rng.integers(0, seq - 256 + 1))
        g0 = (b * heads + h) * seq + t0
        ref, refabs = eo.attn_scores(om, t.blocks[g0:g0 + 256], 1, 1, 256, qpk, q[b, h * qpk:(h + 1) * qpk], 128 ** -0.5)
        check_fused(s[b, h * qpk:(h + 1) * qpk, t0:t0 + 256], ref[0], refabs[0], f"scores q{qpk} full")
    assert np.isfinite(s).all()


def check_full_attn_values(B, eo, t, qpk, n_heads_checked=3):
    batch, heads, seq, _ = t.shape
    om = oracle_meta_from_lib(eo, t.meta)
    rng = np.random.Generator(np.random.PCG64(seq * 3 + qpk))
    scores = (rng.standard_normal((batch, heads * qpk, seq)) * 2.0).astype(np.float32)
    got = gpu_attn_values(B, t.meta, t.blocks, batch, heads, seq, qpk, scores)
    assert np.isfinite(got).all()
    for _ in range(n_heads_checked):
        b, h = int(rng.integers(batch)), int(rng.integers(heads))
        g0 = (b * heads + h) * seq
        ref, refabs = eo.attn_values(om, t.blocks[g0:g0 + seq], 1, 1, seq, qpk, scores[b:b + 1, h * qpk:(h + 1) * qpk])
        check_fused(got[b, h * qpk:(h + 1) * qpk], ref[0], refabs[0], f"values q{qpk} full")


def test_config3_kv_cache_full_size(B, eo, W, synth):
    k, v = W.config3(which=("K", "V"))
    assert k.n_groups == 8 * 32 * 4096
    check_full_decompress(B, eo, k)
    check_full_attn(B, eo, synth, k, 1)
    check_full_decompress(B, eo, v)
    check_full_attn_values(B, eo, v, 1)


def test_config4_llama70b_mlp_full_size(B, eo, W, synth):
    for t in W.config4(names=("gate", "down")):
        assert t.n_groups == 1835008
        om, d_meta, d_blocks = check_full_decompress(B, eo, t)
        check_full_gemv(B, eo, synth, t, om, d_meta, d_blocks, 1)


def test_config5_long_context_gqa_full_size(B, eo, W, synth):
    k, v = W.config5(which=("K", "V"))
    assert k.n_groups == 16 * 8 * 32768
    check_full_decompress(B, eo, k)
    check_full_attn(B, eo, synth, k, 8)
    check_full_attn_values(B, eo, v, 8, n_heads_checked=2)


def test_config4_streams_past_4_gib_of_output(B, eo, W):
    """cfg-4 streams of 1 GiB and 4 GiB (2^24 and 2^26 groups: 4 GiB and 16 GiB of fp16, byte offsets beyond 2^32 and
    TMA row coordinates beyond 2^24), built as bench.py builds them by tiling the encoded gate matrix on the device.
    Compared bit for bit with the oracle: the first and last tile, both sides of every 2^32-byte boundary of the
    output, and 4096 random groups; in between, a hash of every copy of the matrix must equal the first copy's."""
    (t,) = W.config4(names=("gate",))
    om = oracle_meta_from_lib(eo, t.meta)
    d_meta, d_one = B.meta_to_device(t.meta), dev(t.blocks)
    n1 = t.n_groups
    want_one = None
    for log2n in (24, 26):
        n = 1 << log2n
        reps = -(-n // n1)
        d_blocks = d_one.repeat(reps, 1)[:n].contiguous()
        d_out = torch.empty(n * 128, dtype=torch.float16, device="cuda")
        B.ecco_decompress(d_meta, d_blocks, n, d_out)
        torch.cuda.synchronize()
        assert B.ecco_device_status() == 0
        out = d_out.view(n, 128)
        per_4gib = (1 << 32) // 256                         # groups per 2^32 bytes of output
        rng = np.random.Generator(np.random.PCG64(log2n))
        idx = [np.arange(64), np.arange(n - 64, n), rng.integers(0, n, 4096)]
        for b in range(per_4gib, n, per_4gib):
            idx.append(np.arange(b - 64, b + 64))
        idx = np.unique(np.concatenate(idx))
        got = out[torch.from_numpy(idx).cuda()].cpu().numpy()
        assert_bit_exact(got, eo.decode_threads(om, t.blocks[idx % n1], host_threads()))
        # every whole copy of the matrix decodes to the same bits as the first one, which is compared in full
        if want_one is None:
            assert_device_equals_oracle(eo, om, t.blocks, d_out[: n1 * 128])
            want_one = True
        first = out[:n1].view(torch.int16)
        for r in range(1, n // n1):
            assert torch.equal(out[r * n1:(r + 1) * n1].view(torch.int16), first), (log2n, r)
        tail = n - (n // n1) * n1
        if tail:
            assert torch.equal(out[n - tail:].view(torch.int16), first[:tail]), (log2n, "tail")
        del d_blocks, d_out, out, first


# ------------------------------------------------------------------ 2x activation codec
@pytest.mark.parametrize("n_groups", [0, 1, 7, 8, 9, 1000, 4097, 1 << 16])
def test_act2x_compress_and_decompress_match_oracle(B, eo, synth, n_groups):
    x = synth.activations(max(n_groups, 1), 64, 300 + n_groups % 97)[:n_groups]
    if n_groups > 8:
        x[3] = np.float16(-0.75)                     # constant group: zero scale
        x[5] = (x[5].astype(np.float32) * 1000).astype(np.float16)
        x[6] = (x[6].astype(np.float32) * 1e-4).astype(np.float16)   # subnormal-sized steps
    d_x = torch.from_numpy(np.ascontiguousarray(x)).cuda() if n_groups else torch.empty(64, dtype=torch.float16, device="cuda")
    d_blocks = torch.full((max(n_groups, 1), 64), 0xEE, dtype=torch.uint8, device="cuda")
    B.ecco_act_compress(d_x, n_groups, d_blocks)
    d_out = torch.empty((max(n_groups, 1), 64), dtype=torch.float16, device="cuda")
    B.ecco_act_decompress(d_blocks, n_groups, d_out)
    torch.cuda.synchronize()
    if n_groups == 0:
        return
    want_blocks = eo.act_encode(x)
    got_blocks = d_blocks.cpu().numpy()
    bad = np.nonzero((got_blocks != want_blocks).any(axis=1))[0]
    assert bad.size == 0, f"{bad.size} blocks differ, first {bad[:4]}"
    assert np.array_equal(d_out.cpu().numpy().view(np.uint16), eo.act_decode(want_blocks).view(np.uint16))
    # decompression is total: random bytes decode like the oracle says
    rb = synth.random_blocks(n_groups, 17)
    d_rb = torch.from_numpy(rb).cuda()
    B.ecco_act_decompress(d_rb, n_groups, d_out)
    torch.cuda.synchronize()
    got, want = d_out.cpu().numpy().view(np.uint16), eo.act_decode(rb).view(np.uint16)
    finite = np.isfinite(eo.act_decode(rb).astype(np.float32))       # NaN payloads may differ, everything else may not
    assert np.array_equal(got[finite], want[finite])


@pytest.mark.parametrize("loads,past", [(1, 0), (1, 1), (2, 0), (2, 1), (4, 0), (4, 1)])
def test_act2x_at_the_change_of_loads_per_thread(B, eo, synth, loads, past):
    """Multiples of eight CTAs of 256 threads per SM, four threads to a group, whose last CTA is full, and the next call, whose last CTA
    has one group.  The first multiple is the largest call with one load per thread in the compressor, the next call the smallest with two."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    test_act2x_compress_and_decompress_match_oracle(B, eo, synth, sms * 8 * 256 * loads // 4 + past)


# ------------------------------------------------------------------ fused attention output (softmax . V)
def gpu_attn_values(B, lmeta, blocks, batch, heads, seq, qpk, scores):
    d_meta, d_blocks, d_s = B.meta_to_device(lmeta), dev(blocks), dev(scores)
    d_o = torch.full((batch, heads * qpk, 128), float("nan"), dtype=torch.float32, device="cuda")
    wsb = B.ecco_attn_values_workspace_bytes(batch, heads, seq, qpk)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    ws.fill_(0xCD)
    B.ecco_attn_values(d_meta, d_blocks, batch, heads, seq, qpk, d_s, d_o, ws, wsb)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    return d_o.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("batch,heads,seq,qpk", [(2, 4, 256, 1), (2, 4, 256, 8), (1, 3, 77, 4), (1, 1, 1, 1), (2, 2, 1300, 3),
                                                 (1, 2, 5000, 2)])
def test_attn_values_match_oracle(B, eo, kv_small, synth, batch, heads, seq, qpk):
    meta = kv_small["meta"]
    n = batch * heads * seq
    blocks = np.tile(kv_small["blocks"], (-(-n // 2048), 1))[:n]
    rng = np.random.Generator(np.random.PCG64(seq * 7 + qpk))
    scores = (rng.standard_normal((batch, heads * qpk, seq)) * 2.5).astype(np.float32)
    got = gpu_attn_values(B, lib_meta_from_oracle(B, meta), blocks, batch, heads, seq, qpk, scores)
    ref, refabs = eo.attn_values(meta, blocks, batch, heads, seq, qpk, scores)
    check_fused(got, ref, refabs, f"values q{qpk}")


def test_attn_values_on_garbage_blocks_and_peaked_softmax(B, eo, kv_small, synth):
    meta = kv_small["meta"]
    rb = synth.random_blocks(2 * 2 * 700, 321)             # duplicate pad locations, clips, 16-pad groups
    rng = np.random.Generator(np.random.PCG64(5))
    scores = (rng.standard_normal((2, 4, 700)) * 2).astype(np.float32)
    scores[0, 1, :] = -50.0
    scores[0, 1, 333] = 10.0                               # one-hot softmax
    got = gpu_attn_values(B, lib_meta_from_oracle(B, meta), rb, 2, 2, 700, 2, scores)
    ref, refabs = eo.attn_values(meta, rb, 2, 2, 700, 2, scores)
    check_fused(got, ref, refabs, "values q2 garbage")


@pytest.mark.parametrize("qpk", [1, 8])
def test_attn_values_keeps_small_probabilities(B, eo, kv_small, synth, qpk):
    """One token takes almost all the weight and its vector is all zeros, so every output is the sum of the other
    tokens' contributions at p ~ 1e-9: probabilities must survive the trip through the fp16 operands of the tensor
    cores.  A second row spreads its weight evenly over 5000 tokens (p = 2e-4 each, below fp16's normal range).
    Bound: 1e-3 sum p|V| plus 2^-38 sum |V|, the floor of the scaled fp16 pair."""
    meta = kv_small["meta"]
    seq = 5000
    rng = np.random.Generator(np.random.PCG64(17))
    x = synth.kv_cache(1, 1, seq, 1003, 3003).reshape(seq, 128).copy()
    x[1234] = 0
    blocks, _ = eo.encode(meta, x.astype(np.float16), eo.SELECT_MINMAX)
    dec = eo.decode(meta, blocks).astype(np.float64)
    assert not dec[1234].any()
    scores = (rng.standard_normal((1, qpk, seq))).astype(np.float32)
    scores[0, 0, 1234] += 22.0                             # p of the others ~ e^-22 / 1: 3e-10
    if qpk > 1:
        scores[0, 1, :] = 0.25                             # uniform: p = 2e-4 for every token
    got = gpu_attn_values(B, lib_meta_from_oracle(B, meta), blocks, 1, 1, seq, qpk, scores)
    ref, refabs = eo.attn_values(meta, blocks, 1, 1, seq, qpk, scores)
    floor = np.abs(dec).sum(axis=0) * 2.0 ** -38
    err = np.abs(got - ref)
    assert np.all(err <= TOL * refabs + floor), float((err / (TOL * refabs + floor)).max())
    assert np.abs(ref[0, 0]).max() < 1e-6 and np.abs(got[0, 0]).max() > 0      # the small sums are really there
    if qpk > 1:
        assert np.all(err[0, 1] <= 2e-5 * refabs[0, 1])    # evenly spread weights: far inside the bound


# A weight exp(s - m) is off by 2 + 1.2 |s - m| units in the last place at most (the documented bound of __expf), and so is every factor
# that takes sums to a larger maximum.  Weights that count, above 1e-4 of the largest, have |s - m| < 10: 14 units, as much again for the
# factors, 28 * 2^-23 = 3.3e-6; fp32 sums of up to 40 000 terms in chains of some hundred add 2^-24 sqrt(200): 1e-6.  Twice that.  A weight
# below 2^-39 of the largest is lost: the floor.
VALUES_TOL = 1e-5


def values_floor(eo, meta, blocks, batch, heads, seq, qpk):
    dec = np.abs(eo.decode(meta, blocks).astype(np.float64)).reshape(batch, heads, 1, seq, 128).sum(axis=3)
    return 2.0 ** -38 * np.broadcast_to(dec, (batch, heads, qpk, 128)).reshape(batch, heads * qpk, 128)


@pytest.mark.parametrize("batch,heads,seq,qpk", [(1, 1, 31, 8), (1, 1, 6000, 5), (3, 50, 65, 1), (2, 8, 777, 2), (1, 3, 40000, 1), (1, 4, 22000, 8), (2, 70, 590, 3)])
def test_attn_values_of_every_unit_size(B, eo, kv_small, batch, heads, seq, qpk):
    """Units of one warp to nineteen, one or two of them to a CTA; one head in a piece per SM; more short heads than SMs."""
    meta = kv_small["meta"]
    n = batch * heads * seq
    blocks = np.tile(kv_small["blocks"], (-(-n // 2048), 1))[:n]
    scores = (np.random.Generator(np.random.PCG64(seq)).standard_normal((batch, heads * qpk, seq)) * 3).astype(np.float32)
    got = gpu_attn_values(B, lib_meta_from_oracle(B, meta), blocks, batch, heads, seq, qpk, scores)
    ref, refabs = eo.attn_values(meta, blocks, batch, heads, seq, qpk, scores)
    check_fused(got, ref, refabs, "values unit sizes", VALUES_TOL, values_floor(eo, meta, blocks, batch, heads, seq, qpk))


@pytest.mark.parametrize("batch,heads,seq,qpk", [(8, 295, 20, 4), (3, 100, 33, 8), (9, 50, 65, 2), (4, 128, 150, 3), (10, 26, 513, 8)])
def test_attn_values_of_many_short_rows(B, eo, kv_small, batch, heads, seq, qpk):
    """Teams of one to eight warps with heads of their own, up to sixteen teams to a CTA; rows that end inside a tile and a turn."""
    test_attn_values_of_every_unit_size(B, eo, kv_small, batch, heads, seq, qpk)


@pytest.mark.parametrize("batch,heads,seq,qpk", [(16, 32, 300, 2), (4, 32, 1500, 1)])
def test_attn_values_error_does_not_grow_with_the_tiles_of_a_warp(B, eo, kv_small, batch, heads, seq, qpk):
    """2-norm of the error over that of the result, rows of which a warp takes three tiles.  An addition is off by 0.43 * 2^-24 of its
    result (rms), a chain of n terms of random sign by that times sqrt(n / 2), 47 tiles one after the other by 1.2e-7.  A weight
    is off by a last place or two (2^-24..2^-22), at random over some hundred tokens that count: 1e-7.  Together 1.6e-7 at most; sums
    that grow inside the tensor cores, which cut off, are off by 2.5e-7 here.  Limit 2e-7."""
    n = batch * heads * seq
    blocks = np.tile(kv_small["blocks"], (-(-n // 2048), 1))[:n]
    scores = np.random.Generator(np.random.PCG64(seq)).standard_normal((batch, heads * qpk, seq)).astype(np.float32)
    got = gpu_attn_values(B, lib_meta_from_oracle(B, kv_small["meta"]), blocks, batch, heads, seq, qpk, scores)
    dec = np.tile(eo.decode(kv_small["meta"], kv_small["blocks"]), (-(-n // 2048), 1))[:n].astype(np.float64).reshape(batch * heads, seq, 128)
    p = np.exp(scores.astype(np.float64).reshape(batch * heads, qpk, seq))
    ref = np.matmul(p / p.sum(axis=-1, keepdims=True), dec).reshape(got.shape)
    rel = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    assert rel <= 2e-7, rel


def values_plan(heads, seq):
    """(warps of a unit, teams) that ecco_attn_values takes: the rule of av_teams (ecco_kernels.cu) restated, to see what a shape exercises."""
    tiles, ctas = (seq + 31) // 32, torch.cuda.get_device_properties(0).multi_processor_count
    ctas = min(ctas, 256, heads * tiles)
    best = None
    for w in range(19, 0, -1):
        cost = -(-heads * -(-tiles // w) // ctas) * (6 + w) + max(1, -(-heads // ctas) - 1) * 10
        cost += cost // 32 + 1 if w > 16 else 0
        if best is None or cost < best[0]:
            best = (cost, w, 1)
    for t in range(2, 17):
        for w in range(1, 16 // t + 1):
            cost = -(-heads // (ctas * t)) * (-(-tiles // w) * (6 + w * min(t, -(-heads // ctas))) + 10)
            if cost < best[0]:
                best = (cost, w, t)
    return best[1:]


@pytest.mark.parametrize("heads,seq,qpk,plan", [(296, 4096, 3, (16, 1)), (160, 7777, 2, (19, 1)), (300, 512, 8, (4, 3))])
def test_attn_values_with_many_tiles_of_a_row_to_a_warp(B, eo, kv_small, heads, seq, qpk, plan):
    """Rows of which a warp takes four to thirteen tiles one after the other, in both kernels and in teams: random scores, held to
    the 2-norm limit above, too; scores that grow or fall along the row, so that every tile or only the first raises the maximum; rows whose first
    half is masked, so that warps go from tiles without any weight to others."""
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert values_plan(heads, seq) == plan and -(-seq // (32 * plan[0])) >= 4
    meta, n = kv_small["meta"], heads * seq
    blocks = np.tile(kv_small["blocks"], (-(-n // 2048), 1))[:n]
    dec = eo.decode(meta, kv_small["blocks"]).astype(np.float64)
    s = np.random.Generator(np.random.PCG64(seq)).standard_normal((heads, qpk, seq)).astype(np.float32)
    ramp = np.linspace(-60, 60, seq, dtype=np.float32)
    s[1::4] += ramp
    s[2::4] -= ramp
    s[3::4, :, : seq // 2] = -np.inf
    got = gpu_attn_values(B, lib_meta_from_oracle(B, meta), blocks, 1, heads, seq, qpk, s.reshape(1, heads * qpk, seq)).reshape(heads, qpk, 128)
    p = np.exp(s.astype(np.float64) - s.max(axis=2, keepdims=True))
    p /= p.sum(axis=2, keepdims=True)
    # blocks repeat after 2048 groups: weights of the same block are added first
    at = (np.arange(n).reshape(heads, seq)) % 2048
    folded = np.stack([np.stack([np.bincount(at[h], p[h, q], 2048) for q in range(qpk)]) for h in range(heads)])
    ref, refabs = folded @ dec, folded @ np.abs(dec)
    floor = 2.0 ** -38 * np.stack([np.bincount(at[h], minlength=2048) @ np.abs(dec) for h in range(heads)])[:, None]
    check_fused(got, ref, refabs, "values many tiles", VALUES_TOL, floor)
    rel = float(np.linalg.norm(got[::4] - ref[::4]) / np.linalg.norm(ref[::4]))
    assert rel <= 2e-7, rel


@pytest.mark.parametrize("seq", [33, 700, 3000])
def test_attn_values_with_rising_scores_and_any_workspace(B, eo, kv_small, seq):
    """Scores that grow along the row, fall, or hold their largest value in the last token, over heads split between several blocks, each of
    which has one unit of its head (several: the test above); the same bits whatever the workspace held."""
    meta, heads, qpk = kv_small["meta"], 3, 4
    rng = np.random.Generator(np.random.PCG64(seq))
    n = heads * seq
    blocks = np.tile(kv_small["blocks"], (-(-n // 2048), 1))[:n]
    s = (rng.standard_normal((1, heads * qpk, seq)) * 2).astype(np.float32)
    s[0, 0::4] += np.linspace(-60, 60, seq, dtype=np.float32)
    s[0, 1::4] += np.linspace(60, -60, seq, dtype=np.float32)
    s[0, 2::4, -1] = 80.0
    d_meta, d_blocks, d_s = B.meta_to_device(lib_meta_from_oracle(B, meta)), dev(blocks), dev(s)
    wsb = B.ecco_attn_values_workspace_bytes(1, heads, seq, qpk)
    first = None
    for fill in (0, 0xFF, 0x3C, "left"):
        if fill != "left":
            ws = torch.full((wsb,), fill, dtype=torch.uint8, device="cuda")
        out = torch.full((1, heads * qpk, 128), float("nan"), dtype=torch.float32, device="cuda")
        B.ecco_attn_values(d_meta, d_blocks, 1, heads, seq, qpk, d_s, out, ws, wsb)
        first = out if first is None else first
        assert torch.equal(out, first), fill
    ref, refabs = eo.attn_values(meta, blocks, 1, heads, seq, qpk, s)
    check_fused(first.cpu().numpy().astype(np.float64), ref, refabs, "values rising", VALUES_TOL, values_floor(eo, meta, blocks, 1, heads, seq, qpk))


@pytest.mark.parametrize("seq", [301, 4100])
def test_attn_values_with_masked_scores(B, eo, kv_small, synth, seq):
    """Scores of -inf (masked tokens) carry no weight: at the start of a row (before the row statistics have seen any
    finite score), in the middle, in whole 16-byte chunks and at a ragged end; rows of odd length start at addresses
    that are not 16-byte aligned."""
    meta = kv_small["meta"]
    heads, qpk = 2, 3
    n = heads * seq
    blocks = np.tile(kv_small["blocks"], (-(-n // 2048), 1))[:n]
    rng = np.random.Generator(np.random.PCG64(5 + seq))
    scores = (rng.standard_normal((1, heads * qpk, seq)) * 2.0).astype(np.float32)
    scores[0, :, :9] = -np.inf
    scores[0, 1, 100:164] = -np.inf
    scores[0, 2, -3:] = -np.inf
    scores[0, 3, rng.random(seq) < 0.5] = -np.inf
    scores[0, 4, 1:] = -np.inf
    scores[0, 4, 0] = 0.5                                  # a single live token, first in the row
    got = gpu_attn_values(B, lib_meta_from_oracle(B, meta), blocks, 1, heads, seq, qpk, scores)
    ref, refabs = eo.attn_values(meta, blocks, 1, heads, seq, qpk, scores)
    assert np.isfinite(ref).all()
    check_fused(got, ref, refabs, "values masked")


# ------------------------------------------------------------------ online KV compressor
def gpu_kv_compress(B, lmeta, x):
    n = x.size // 128
    d_meta = B.meta_to_device(lmeta)
    d_x = dev(x.reshape(-1)) if n else torch.empty(128, dtype=torch.float16, device="cuda")
    d_blocks = torch.full((max(n, 1), 64), 0xEE, dtype=torch.uint8, device="cuda")
    B.ecco_kv_compress(d_meta, d_x, n, d_blocks)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    return d_blocks.cpu().numpy()[:n]


def assert_blocks_equal(got, want):
    bad = np.nonzero((got != want).any(axis=1))[0]
    assert bad.size == 0, f"{bad.size} of {got.shape[0]} blocks differ; first {bad[:5]}"


@pytest.mark.parametrize("n_groups", [0, 1, 7, 8, 9, 2048])
def test_kv_compress_matches_oracle_encoder(B, eo, kv_small, n_groups):
    meta = kv_small["meta"]
    x = kv_small["k"].reshape(-1, 128)[:n_groups]
    got = gpu_kv_compress(B, lib_meta_from_oracle(B, meta), x)
    if n_groups:
        assert_blocks_equal(got, kv_small["blocks"][:n_groups])


def test_kv_compress_edge_groups_and_s16(B, eo, kv_small, synth):
    meta = kv_small["meta"]
    rng = np.random.Generator(np.random.PCG64(77))
    groups = [np.zeros(128), np.full(128, 0.5), np.full(128, -3.0), np.concatenate([np.full(64, 1.0), np.full(64, -1.0)]),
              np.full(128, 2.0 ** -24), rng.standard_normal(128) * 1e-3, rng.standard_normal(128) * 300,   # saturating scales
              np.where(np.arange(128) % 2 == 0, 5.0, -5.0), np.arange(128) - 64.0, rng.choice([-2.0, 0.0, 2.0], 128)]
    for _ in range(200):
        g = rng.standard_normal(128) * rng.choice([0.1, 1.0, 10.0])
        g[rng.integers(128)] *= rng.choice([1.0, 20.0])
        if rng.random() < 0.3:
            g[rng.integers(128, size=5)] = g[rng.integers(128)]            # ties in |x|
        groups.append(g)
    x = np.array(groups, dtype=np.float16)
    want, st = eo.encode(meta, x, eo.SELECT_MINMAX)
    assert st.clipped_groups > 0 and st.padded_groups > 0
    assert_blocks_equal(gpu_kv_compress(B, lib_meta_from_oracle(B, meta), x), want)
    # the paper's hardware compressor works with 16 patterns
    cal = synth.kv_cache(1, 4, 512, 2003, 3003)
    m16 = eo.calibrate(cal, S=16, H=4, seed=3, select=eo.SELECT_MINMAX)
    want, _ = eo.encode(m16, kv_small["k"], eo.SELECT_MINMAX)
    assert_blocks_equal(gpu_kv_compress(B, lib_meta_from_oracle(B, m16), kv_small["k"]), want)
    # a skewed codebook: long streams (heavy clipping) and short ones (16 pads)
    skew = make_meta(eo, skew_lens, seed=3)
    xs = (rng.standard_t(3, size=(512, 128)) * 0.05).astype(np.float16)
    want, st = eo.encode(skew, xs, eo.SELECT_MINMAX)
    assert_blocks_equal(gpu_kv_compress(B, lib_meta_from_oracle(B, skew), xs), want)


@pytest.mark.parametrize("kind,n_groups", [("calibrated", 16383), ("calibrated", 16384), ("s16", 16385), ("equal centroids", 16386),
                                           ("dense centroids", 16387), ("wide centroids", 16384), ("skewed codes", 16385),
                                           ("midpoint at zero", 16386)])
def test_kv_compress_of_many_groups_matches_the_host_encoder(B, eo, kv_small, synth, kind, n_groups):
    """Calls on both sides of the size from which eight lanes share a group, ragged in the last four groups, on groups that
    decide at the edges: values at midpoints of centroids, ties, zeros, one value only, saturating and subnormal scales,
    patterns with equal centroids, with several midpoints per table cell (a zero the first of them, too) and with centroids far outside [-1, 1]."""
    rng = np.random.Generator(np.random.PCG64(n_groups))
    if kind == "calibrated":
        om = kv_small["meta"]
    elif kind == "s16":
        om = eo.calibrate(synth.kv_cache(1, 4, 512, 2003, 3003), S=16, H=4, seed=3, select=eo.SELECT_MINMAX)
    else:
        om = make_meta(eo, skew_lens, S=7, e=-3, seed=5)
        for k in range(om.S):
            p = np.sort(rng.uniform(-1, 1, 15))
            if kind == "equal centroids":
                p[3:6], p[9] = p[3], p[10]
            elif kind == "dense centroids":
                p[2:12] = p[2] + np.arange(10) * 0.0007
            elif kind == "wide centroids":
                p *= 4.0
            elif kind == "midpoint at zero":
                p = np.concatenate([np.linspace(-0.9, -0.1, 7), [-0.0003, 0.0003, 0.0011], np.linspace(0.2, 0.9, 5)])
            for j, c in enumerate(np.sort(p.astype(np.float16)).view(np.uint16)):
                om.pattern[k][j] = int(c)
    lm = lib_meta_from_oracle(B, om)
    pat = om.patterns()[: om.S].astype(np.float64)
    x = synth.kv_cache(1, 4, (n_groups + 3) // 4, 41, 42).reshape(-1, 128)[:n_groups].copy()
    for g in range(0, n_groups, 11):                       # values at (or next to) midpoints of a pattern, abs-max a power of two
        p = pat[g % om.S]
        mids = 0.5 * (p[1:] + p[:-1])
        x[g] = (rng.choice(mids, 128) * 4.0).astype(np.float16)
        x[g, rng.integers(128)] = 4.0
    x[1], x[2], x[3], x[5] = 0, 0.5, 2.0 ** -24, np.where(np.arange(128) % 2 == 0, 60000.0, -60000.0)
    x[6] = (rng.standard_normal(128) * 3000).clip(-60000, 60000).astype(np.float16)
    x[7] = (rng.standard_normal(128) * 1e-6).astype(np.float16)
    x[8, :] = rng.choice(np.array([-2.0, 0.0, 2.0], dtype=np.float16), 128)
    want, _ = B.ecco_encode_host(lm, x, B.SELECT_MINMAX | B.KEEP_EXPONENT)
    assert_blocks_equal(gpu_kv_compress(B, lm, x), want)


def test_kv_compress_of_many_groups_maps_a_second_infinity_to_an_end_centroid(B, eo):
    """Blocks of groups with infinities are unspecified, but only the abs-max itself carries the abs-max's symbol: a value above all midpoints
    takes the last centroid, one below all of them the first.  Codewords of four bits, so that every group is cut off and no outlier hides the symbol."""
    om = make_meta(eo, lambda k, h, rng: [4] * 16, S=5, e=-3, seed=6)
    x = np.zeros((16384, 128), dtype=np.float16)
    x[::3, :3] = np.inf, np.inf, -np.inf
    x[1::3, 5:8] = -np.inf, -np.inf, np.inf
    dec = eo.decode(om, gpu_kv_compress(B, lib_meta_from_oracle(B, om), x)).astype(np.float64)
    scale, ends = 448.0 * 2.0 ** om.e, om.patterns()[0].astype(np.float64)[[0, 14]]      # no pattern fits: the first one
    first, last = np.float16(scale * ends)
    assert (dec[::3, :3] == [scale, last, first]).all() and (dec[1::3, 5:8] == [-scale, first, last]).all()


def test_kv_compress_full_size_round_trip(B, eo, W, synth):
    """cfg 3 K cache: GPU-compressed blocks equal the host encoder's, and decompress to the same fp16."""
    (t,) = W.config3(which=("K",), keep_source=True)
    got = gpu_kv_compress(B, t.meta, t.source)
    assert_blocks_equal(got, t.blocks)


# ------------------------------------------------------------------ variable-length container
def oracle_offsets_from_index(index, n):
    nc = (n + 4095) // 4096
    idx64 = index[: 8 * (1 + nc)].view(np.uint64)
    off32 = index[8 * (1 + nc): 8 * (1 + nc) + 4 * n].view(np.uint32)
    return np.concatenate([idx64[1:][np.arange(n) >> 12] + off32, idx64[:1]]).astype(np.uint64)


def gpu_var_decompress(B, lmeta, stream, index, n):
    d_out = torch.full((n, 128), float("nan"), dtype=torch.float16, device="cuda")
    B.ecco_var_decompress(B.meta_to_device(lmeta), dev(stream), dev(index), n, d_out)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    return d_out.cpu().numpy()


@pytest.mark.parametrize("n_groups", [1, 31, 33, 1000, 2048])
def test_var_decompress_matches_oracle(B, eo, cfg1_small, n_groups):
    meta = cfg1_small["meta"]
    lm = lib_meta_from_oracle(B, meta)
    x = cfg1_small["w"].reshape(-1, 128)[:n_groups]
    stream, index, total = B.ecco_var_encode_host(lm, x, B.SELECT_MSE | B.KEEP_EXPONENT)
    got = gpu_var_decompress(B, lm, stream, index, n_groups)
    assert_bit_exact(got, eo.var_decode(meta, stream, oracle_offsets_from_index(index, n_groups)))


def test_var_decompress_is_total_on_garbage(B, eo, cfg1_small, synth):
    """Random stream bytes with a valid-looking but arbitrary index: overlapping, empty and over-long groups."""
    meta = cfg1_small["meta"]
    lm = lib_meta_from_oracle(B, meta)
    n = 4096 + 100
    rng = np.random.Generator(np.random.PCG64(12))
    stream = synth.random_blocks(4096, 5).reshape(-1)                      # 256 KiB of noise, a multiple of 16
    total = stream.size * 8 - 37
    starts = np.sort(rng.integers(0, total, n)).astype(np.uint64)
    starts[5] = starts[4]                                                   # empty group
    nc = (n + 4095) // 4096
    index = np.zeros((8 * (1 + nc) + 4 * n + 15) // 16 * 16, dtype=np.uint8)
    idx64 = index[: 8 * (1 + nc)].view(np.uint64)
    idx64[0] = total
    for c in range(nc):
        idx64[1 + c] = starts[c * 4096]
    index[8 * (1 + nc): 8 * (1 + nc) + 4 * n].view(np.uint32)[:] = (starts - idx64[1:][np.arange(n) >> 12]).astype(np.uint32)
    got = gpu_var_decompress(B, lm, stream, index, n)
    assert_bit_exact(got, eo.var_decode(meta, stream, np.concatenate([starts, [np.uint64(total)]]).astype(np.uint64)))


@pytest.mark.parametrize("long_share", [0.0, 0.03, 1.0])
def test_var_decompress_groups_longer_than_a_lane_holds(B, eo, cfg1_small, synth, long_share):
    """A lane stages 640 bits of the stream; longer groups (values from the rare, long codewords of the ends of the range) are
    fetched in two parts, in some lanes of a warp or in all.  Exact: decoding has one result."""
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    n = 1000 + 7
    rng = np.random.Generator(np.random.PCG64(31))
    w = synth.weight_matrix(128, 1024, 9).reshape(-1, 128)[:n].astype(np.float32)
    ends = rng.choice([-1.0, 1.0], (n, 128)) * rng.uniform(0.6, 1.0, (n, 128)) * np.abs(w).max(1, keepdims=True)
    x = np.where(rng.random((n, 1)) < long_share, ends, w).astype(np.float16)
    stream, index, total = B.ecco_var_encode_host(lm, x, B.SELECT_MSE | B.KEEP_EXPONENT)
    offs = oracle_offsets_from_index(index, n).astype(np.int64)
    covered = np.diff(offs) + offs[:n] % 64
    assert (covered > 640).mean() >= 0.4 * long_share
    got = gpu_var_decompress(B, lm, stream, index, n)
    assert_bit_exact(got, eo.var_decode(cfg1_small["meta"], stream, oracle_offsets_from_index(index, n)))


def test_var_decompress_config2_gate_full_size(B, eo, W, synth):
    (t,) = W.config2(names=("gate",), keep_source=True)
    stream, index, total = B.ecco_var_encode_host(t.meta, t.source, B.SELECT_MSE | B.KEEP_EXPONENT)
    n = t.n_groups
    d_out = torch.empty((n, 128), dtype=torch.float16, device="cuda")
    B.ecco_var_decompress(B.meta_to_device(t.meta), dev(stream), dev(index), n, d_out)
    torch.cuda.synchronize()
    om = oracle_meta_from_lib(eo, t.meta)
    offs = oracle_offsets_from_index(index, n)
    # sampled runs of consecutive groups (the oracle needs each group's end = the next group's start)
    rng = np.random.Generator(np.random.PCG64(2))
    for g0 in [0, n - 512] + [int(v) for v in rng.integers(0, n - 512, 6)]:
        want = eo.var_decode(om, stream, np.concatenate([offs[g0:g0 + 512], offs[g0 + 512:g0 + 513]]))
        assert_bit_exact(d_out[g0:g0 + 512].cpu().numpy(), want)
    assert bool(torch.isfinite(d_out).all())
    assert total / n < 512                                                  # on average the stream is shorter than the blocks


# ------------------------------------------------------------------ capture into a CUDA graph
def test_calls_can_be_captured_into_a_cuda_graph(B, eo, kv_small, cfg1_small, synth):
    """The device calls neither synchronise nor allocate, so a chain of them can be captured into a CUDA graph
    (after one eager call of each, which sets the kernels' attributes) and replayed; the replay gives the eager
    results bit for bit, also after the inputs have changed in place."""
    wm, km = B.meta_to_device(lib_meta_from_oracle(B, cfg1_small["meta"])), B.meta_to_device(lib_meta_from_oracle(B, kv_small["meta"]))
    wb, kb = dev(cfg1_small["blocks"]), dev(kv_small["blocks"])                 # 256 x 1024 weights, K cache [2][4][256]
    n_out, k, heads, seq, qpk = 256, 1024, 8, 256, 2
    x = dev(synth.activations(8, k, 3))
    q = dev(synth.queries(1, heads * qpk, 4))
    out = torch.empty(2048 * 128, dtype=torch.float16, device="cuda")
    y1, y8 = torch.empty((1, n_out), dtype=torch.float32, device="cuda"), torch.empty((8, n_out), dtype=torch.float32, device="cuda")
    sc = torch.empty((1, heads * qpk, seq), dtype=torch.float32, device="cuda")
    av = torch.empty((1, heads * qpk, 128), dtype=torch.float32, device="cuda")
    items1, items8 = [(wm, wb, n_out, k, x, y1)], [(wm, wb, n_out, k, x, y8)]
    nb1, nb8 = B.ecco_gemv_batch_workspace_bytes(items1, 1), B.ecco_gemv_batch_workspace_bytes(items8, 8)
    ws1, ws8 = torch.empty(nb1, dtype=torch.uint8, device="cuda"), torch.empty(nb8, dtype=torch.uint8, device="cuda")
    nbv = B.ecco_attn_values_workspace_bytes(1, heads, seq, qpk)
    wsv = torch.empty(nbv, dtype=torch.uint8, device="cuda")
    a1, a8 = B.gemv_items(items1), B.gemv_items(items8)

    def chain(st):
        B.ecco_decompress(wm, wb, 2048, out, st)
        B.ecco_gemv_batch(a1, 1, ws1, nb1, st)
        B.ecco_gemv_batch(a8, 8, ws8, nb8, st)
        B.ecco_attn_scores(km, kb, 1, heads, seq, qpk, q, 0.0884, sc, st)
        B.ecco_attn_values(km, kb, 1, heads, seq, qpk, sc, av, wsv, nbv, st)

    results = lambda: [t.clone() for t in (out, y1, y8, sc, av)]
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        chain(st)                                          # eager: also the first call of every kernel
        st.synchronize()
        want = results()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            chain(st)
        for t in (out, y1, y8, sc, av):
            t.fill_(float("nan"))
        g.replay()
        st.synchronize()
        assert B.ecco_device_status() == 0
        assert all(torch.equal(a, b) for a, b in zip(want, results()))
        x.mul_(0.5)                                        # new inputs in the same buffers
        q.mul_(2.0)
        g.replay()
        st.synchronize()
        replayed = results()
        chain(st)
        st.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(replayed, results()))
        assert not torch.equal(replayed[1], want[1])


# ------------------------------------------------------------------ stream order of back-to-back calls
def test_back_to_back_calls_keep_stream_order(B, eo, kv_small, cfg1_small, synth):
    """The kernels are launched so that one may start while its predecessor in the stream drains.  Calls that
    depend on each other through a buffer (write-after-write on an output, read-after-write on blocks, scores and
    a shared workspace), issued with no synchronisation in between, must give what they give one at a time."""
    meta, lm = kv_small["meta"], lib_meta_from_oracle(B, kv_small["meta"])
    d_meta = B.meta_to_device(lm)
    reps = 96                                              # 196 608 groups: every SM busy, tails overlap heads
    x = np.tile(kv_small["k"].reshape(-1, 128), (reps, 1))
    n = x.shape[0]
    want_blocks = np.tile(kv_small["blocks"], (reps, 1))
    want_a = np.tile(eo.decode(meta, kv_small["blocks"]), (reps, 1))
    other = np.ascontiguousarray(want_blocks[::-1])        # a second, different tensor of the same size
    want_b = np.ascontiguousarray(want_a[::-1])
    d_x, d_other = dev(x.reshape(-1)), dev(other)
    d_blocks = torch.full((n, 64), 0xEE, dtype=torch.uint8, device="cuda")
    d_out = torch.zeros(n * 128, dtype=torch.float16, device="cuda")
    d_out2 = torch.zeros(n * 128, dtype=torch.float16, device="cuda")
    for _ in range(6):
        B.ecco_kv_compress(d_meta, d_x, n, d_blocks)       # blocks written ...
        B.ecco_decompress(d_meta, d_blocks, n, d_out2)     # ... and read by the next kernel
        B.ecco_decompress(d_meta, d_other, n, d_out)       # the same output twice: the later call wins
        B.ecco_decompress(d_meta, d_blocks, n, d_out)
        B.ecco_decompress(d_meta, d_other, n, d_out)
        d_blocks_snapshot = d_blocks.clone()
        d_blocks.fill_(0xEE)                               # a non-library kernel in between
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    assert_blocks_equal(d_blocks_snapshot.cpu().numpy(), want_blocks)
    assert_bit_exact(d_out2.cpu().numpy().reshape(n, 128), want_a)
    assert_bit_exact(d_out.cpu().numpy().reshape(n, 128), want_b)

    # two products through ONE workspace, then scores -> softmax . V, all back to back
    wmeta, wlm = cfg1_small["meta"], lib_meta_from_oracle(B, cfg1_small["meta"])
    d_wmeta = B.meta_to_device(wlm)
    n_out, k = 4096, 2048
    blocks_a = np.tile(cfg1_small["blocks"], (32, 1))[: n_out * k // 128]
    blocks_b = np.ascontiguousarray(blocks_a[::-1])
    d_a, d_b = dev(blocks_a), dev(blocks_b)
    for batch in (1, 8):
        xs = synth.activations(batch, k, 400 + batch)
        d_xs = dev(xs)
        wsb = B.ecco_gemv_workspace_bytes(n_out, k, batch)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        ws.fill_(0xA5)
        one = []
        for blk in (d_a, d_b):                             # one at a time
            y = torch.empty((batch, n_out), dtype=torch.float32, device="cuda")
            B.ecco_gemv(d_wmeta, blk, n_out, k, d_xs, batch, y, ws, wsb)
            torch.cuda.synchronize()
            one.append(y.cpu().numpy())
        ys = [torch.empty((batch, n_out), dtype=torch.float32, device="cuda") for _ in range(8)]
        for i, y in enumerate(ys):                         # back to back through the same workspace
            B.ecco_gemv(d_wmeta, d_b if i & 1 else d_a, n_out, k, d_xs, batch, y, ws, wsb)
        torch.cuda.synchronize()
        assert B.ecco_device_status() == 0
        for i, y in enumerate(ys):
            assert np.array_equal(y.cpu().numpy(), one[i & 1]), (batch, i)

    batch, heads, seq, qpk = 2, 4, 256, 4
    kb, vb = kv_small["blocks"], np.ascontiguousarray(kv_small["blocks"][::-1])
    q = synth.queries(batch, heads * qpk, 77)
    d_k, d_v, d_q = dev(kb), dev(vb), dev(q)
    wsb = B.ecco_attn_values_workspace_bytes(batch, heads, seq, qpk)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    sc = torch.empty((batch, heads * qpk, seq), dtype=torch.float32, device="cuda")
    out = torch.empty((batch, heads * qpk, 128), dtype=torch.float32, device="cuda")
    B.ecco_attn_scores(d_meta, d_k, batch, heads, seq, qpk, d_q, 0.0884, sc)
    torch.cuda.synchronize()
    B.ecco_attn_values(d_meta, d_v, batch, heads, seq, qpk, sc, out, ws, wsb)
    torch.cuda.synchronize()
    want = out.cpu().numpy().copy()
    for _ in range(4):
        sc.zero_()
        out.zero_()
        B.ecco_attn_scores(d_meta, d_k, batch, heads, seq, qpk, d_q, 0.0884, sc)
        B.ecco_attn_values(d_meta, d_v, batch, heads, seq, qpk, sc, out, ws, wsb)
    torch.cuda.synchronize()
    assert B.ecco_device_status() == 0
    assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("batch", [1, 8])
def test_a_refused_call_keeps_the_stream_order_of_its_neighbours(B, eo, cfg1_small, synth, batch):
    """A grouped product over matrices with different tables ends without doing anything, on SMs that the call before it leaves
    free.  The call behind it must still find that call's output complete: as it does with a synchronisation in between."""
    lm = lib_meta_from_oracle(B, cfg1_small["meta"])
    S, e, pat, cb, kp = lm.tables()
    cb = cb.copy()
    cb[0, 0] = cb[0, 0][::-1]
    d_meta, other = B.meta_to_device(lm), B.meta_to_device(B.ecco_meta_create(S, e, pat, cb, kp))
    d_blocks, n = dev(cfg1_small["blocks"]), 2048          # 64 tiles of 32 groups: 64 SMs
    d_x, d_y = dev(synth.activations(batch, 1024, 5)), torch.zeros((2, batch, 256), device="cuda")
    items = [(d_meta, d_blocks, 256, 1024, d_x, d_y[0]), (other, d_blocks, 256, 1024, d_x, d_y[1])]
    wsb = B.ecco_gemv_batch_workspace_bytes(items, batch)
    ws, arr = torch.empty(wsb, dtype=torch.uint8, device="cuda"), B.gemv_items(items)
    out, act = torch.zeros(n * 128, dtype=torch.float16, device="cuda"), torch.zeros((2 * n, 64), dtype=torch.uint8, device="cuda")
    want = dev(eo.act_encode(eo.decode(cfg1_small["meta"], cfg1_small["blocks"]).reshape(-1)))

    def chain(st):
        B.ecco_decompress(d_meta, d_blocks, n, out, st)
        B.ecco_gemv_batch(arr, batch, ws, wsb, st)
        B.ecco_act_compress(out, 2 * n, act, st)

    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        chain(st)
        st.synchronize()
        assert torch.equal(act, want) and B.ecco_device_status() == B.ERR_INVALID_ARG
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            chain(st)
        for i in range(40):                                # eager and as a graph, whose launches follow one another at once
            out.zero_()
            act.zero_()
            g.replay() if i & 1 else chain(st)
            st.synchronize()
            assert torch.equal(act, want), i
    assert B.ecco_device_status() == B.ERR_INVALID_ARG and not d_y.any()
