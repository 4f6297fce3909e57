"""The kernels for several rows at the sizes where they change: edges of tiles, cells, chunks and panels.

Linears over cells: exact products, summed in fp32.  A product goes through one step of the tensor core, which truncates sixteen of
them to within 2^-22 of S = sum |w x|, then through three additions in its cell, at most sixteen over a warp's cells and four over
warps and CTAs, each rounded to within 2^-24 of S: |y - ref| <= 27 * 2^-24 S < 2e-6 S.  (A lost weight is S / K and more, 1e-4 S at
the longest row here.)  The strips and the LM head add along longer chains, whose errors cancel: they are held to the same.  bf16
outputs add their rounding, 2^-8 |y|.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import decoder_oracle as do
from oracle import oracle
from paper_2504_08838_b200 import binding as sd2
from paper_2504_08838_b200 import synth
from tests.test_gpu_parity import _read_u16

pytestmark = pytest.mark.gpu


def dev(bits):
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int16).copy()).cuda().view(torch.bfloat16)


def bits_of(t):
    return t.view(torch.int16).cpu().numpy().view(np.uint16)


def values(bits):
    return synth.bf16_bits_to_f32(bits).astype(np.float64)


def linear_close(y, W, mask, x, f32):
    ref, S = oracle.masked_linear(W, mask, x)
    tol = 2e-6 * S
    assert np.all(np.abs(y - ref) <= tol + (0.0 if f32 else 2.0 ** -8 * (np.abs(ref) + tol)))


@pytest.mark.parametrize("M,K,N,density,shift", [
    (1, 8, 4, 0.5, 0), (15, 40, 5, 0.5, 0),                          # one cell: one CTA of a cluster has it all
    (17, 129, 8, 0.5, 0), (16, 256, 9, 0.5, 0), (100, 257, 16, 0.5, 0),   # a column, a cell for the second CTA; both panel widths
    (333, 1000, 17, 0.3, 0), (200, 2048, 32, 0.5, 0), (64, 1536, 33, 0.7, 0), (50, 4608, 20, 0.5, 0),   # wide panels, two launches
    (3000, 640, 4, 0.5, 0), (2500, 1152, 12, 0.1, 0),                # five and nine cells a tile: turns of two tiles, of one and a rest
    (200, 4096, 8, 0.5, 0), (200, 4100, 8, 0.5, 0), (1531, 8192, 16, 0.5, 0),  # whole tiles to a group, thirds of tiles
    (77, 3001, 5, 0.5, 0), (77, 3000, 7, 0.5, 1), (40, 1003, 16, 0.9, 3), (9, 5, 6, 1.0, 1),   # rows that do not start on 16 bytes
    (320, 2048, 8, 0.0, 0), (320, 2048, 8, 1.0, 0),                  # nothing kept, everything kept
    (512, 2048, 2, 0.5, 0), (512, 2048, 3, 0.5, 0),                  # the smallest panels of large weights
])
def test_linear_over_cells(M, K, N, density, shift):
    W = synth.normal_bf16(M + K, (M, K), 0.02)
    mask = synth.bernoulli_mask(M + K + 1, (M, K), density) if 0.0 < density < 1.0 else np.full((M, K), int(density), np.uint8)
    x = synth.normal_bf16(M + K + 2, (N, K), 1.0)
    f32 = N % 2 == 0
    h = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4, sd2.SD2_DTYPE_F32 if f32 else sd2.SD2_DTYPE_BF16)
    store = torch.zeros(N * K + shift, dtype=torch.bfloat16, device="cuda")
    store[shift:] = dev(x).view(-1)
    guard = 40
    buf = torch.full((N * M + 2 * guard,), float("nan"), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    sd2.sd2_spmm(h, store[shift:].view(N, K), buf[guard:guard + N * M].view(N, M))
    sd2.sd2_stream_check()
    out = buf.float().cpu().numpy().astype(np.float64)
    assert np.isnan(out[:guard]).all() and np.isnan(out[-guard:]).all() and not np.isnan(out[guard:-guard]).any()
    linear_close(out[guard:-guard].reshape(N, M), W, mask, x, f32)
    sd2.sd2_free(h)


@pytest.mark.parametrize("M,K", [(64, 640), (200, 2048), (96, 3001), (40, 8200)])       # a turn of tiles, whole tiles, unaligned rows, thirds
def test_panels_add_up_like_each_other_and_as_well_as_single_rows(M, K):
    W = synth.normal_bf16(M + K, (M, K), 0.02)
    mask = synth.bernoulli_mask(M + K + 1, (M, K), 0.5)
    x = synth.normal_bf16(M + K + 2, (64, K), 1.0)
    h = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4, sd2.SD2_DTYPE_F32)

    def rows(n):                                                        # all 64 rows in calls of n
        y = torch.full((64, M), float("nan"), dtype=torch.float32, device="cuda")
        for i in range(0, 64, n):
            sd2.sd2_spmm(h, dev(x[i:i + n]), y[i:i + n])
        sd2.sd2_stream_check()
        return y

    panels = rows(4)
    for n in (8, 13, 16, 17, 24, 32, 33, 64):
        assert torch.equal(rows(n), panels), n
    ref, _ = oracle.masked_linear(W, mask, x)

    def error(y):
        return np.linalg.norm(y.double().cpu().numpy() - ref)

    # no further from 64 bits than rows that go alone (chains of mma were 1.2 to 1.7 times as far, truncated sums that they are);
    # a tenth more is left to the draw of 64 M sums
    assert error(panels) <= 1.1 * error(rows(1))
    sd2.sd2_free(h)


@pytest.mark.parametrize("M,K,N", [(40, 100, 4), (77, 3001, 5), (300, 2048, 8), (50, 8200, 16), (200, 2048, 24)])
def test_dropped_weights_take_no_part_whatever_the_activations(M, K, N):
    # infinite and undefined activations reach the rows that keep a weight for them, and no others
    W = synth.normal_bf16(M + K, (M, K), 0.02)
    mask = synth.bernoulli_mask(M + K + 1, (M, K), 0.5)
    x = synth.normal_bf16(M + K + 2, (N, K), 1.0)
    special = [(0, K // 2, 0xFF80), (1, 5, 0x7F80), (1, K - 2, 0x7F80), (2, K - 1, 0x7FC0), (N - 1, 0, 0x7F80), (N - 1, 1, 0xFF80)]
    finite = x.copy()
    for n, k, bits in special:
        x[n, k] = bits
        finite[n, k] = 0
    h = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4, sd2.SD2_DTYPE_F32)
    y = torch.full((N, M), 7.0, dtype=torch.float32, device="cuda")
    sd2.sd2_spmm(h, dev(x), y)
    sd2.sd2_stream_check()
    got = y.double().cpu().numpy()
    extra = np.zeros((N, M))
    with np.errstate(invalid="ignore"):
        for n, k, _ in special:
            extra[n] += np.where(mask[:, k] != 0, values(W[:, k]) * values(x[n:n + 1, k]), 0.0)
    assert np.array_equal(got[~np.isfinite(extra)], extra[~np.isfinite(extra)], equal_nan=True)
    ref, S = oracle.masked_linear(W, mask, finite)
    left = np.isfinite(extra)
    assert left[:3].any() and not left[:3].all() and np.all(np.abs(got - ref)[left] <= 1e-5 * S[left])   # (one sum after the other)
    sd2.sd2_free(h)


def test_dropped_weights_take_no_part_in_a_normalised_row():
    # an infinite column becomes NaN in the norm that is folded into staging: as far as BITMASK handles carry it, and no further
    shape, N, pos = synth.DrafterShape("tiny", 256, 64, 1024, 1), 6, 3
    lin = synth.make_block(2, 0, shape, 0.5)
    x = synth.normal_bf16(70, (N, shape.hidden), 1.0)
    x[2, 100] = 0x7F80
    ones = dev(np.full(shape.hidden, 0x3F80, np.uint16))
    seen = []
    for fmt in (sd2.SD2_FORMAT_BITMASK, sd2.SD2_FORMAT_GAP4):
        hs = [sd2.sd2_compress(W, m, fmt) for W, m in lin]
        kc, vc = (torch.zeros((N, pos + 1, shape.kv), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        ws = torch.zeros(sd2.sd2_decoder_workspace_bytes(hs, N) // 2, dtype=torch.bfloat16, device="cuda")
        y = torch.zeros((N, shape.hidden), dtype=torch.bfloat16, device="cuda")
        sd2.sd2_decoder_block_step(hs, ones, ones, dev(x), y, kc, vc, 8, 2, pos, 1e-5, 1e4, ws)
        sd2.sd2_stream_check()
        seen.append((vc[:, pos].isnan(), y.isnan()))
        for h in hs:
            sd2.sd2_free(h)
    for a, b in zip(*seen):
        assert torch.equal(a, b)
    nans = seen[1][0]
    assert nans[2].any() and not nans[2].all() and not nans[[0, 1, 3, 4, 5]].any()


def test_without_memory_for_cells_the_strips_answer():
    M, K = 600, 2048
    W = synth.normal_bf16(31, (M, K), 0.02)
    mask = synth.bernoulli_mask(32, (M, K), 0.5)
    x = synth.normal_bf16(33, (8, K), 1.0)
    blob = sd2.sd2_pack_host(W, mask, sd2.SD2_FORMAT_GAP4, sd2.SD2_DTYPE_F32)
    sd2.sd2_free(sd2.sd2_load_blob(blob))                               # device set-up is done before counting
    free0 = torch.cuda.mem_get_info()[0]

    def product(h, n):                                                  # all rows in calls of n
        y = torch.full((8, M), float("nan"), dtype=torch.float32, device="cuda")
        for i in range(0, 8, n):
            sd2.sd2_spmm(h, dev(x[i:i + n]), y[i:i + n])
        sd2.sd2_stream_check()
        return y

    def served_by_strips(make, skip):
        sd2.sd2_debug_fail_allocations(skip, 1)
        try:
            h = make()
        except sd2.Sd2Error as e:
            assert e.status == sd2.SD2_ERR_ALLOC
            assert torch.cuda.mem_get_info()[0] == free0
            return "refused"
        finally:
            sd2.sd2_debug_fail_allocations(0, 0)
        y = product(h, 8)
        linear_close(y.double().cpu().numpy(), W, mask, x, True)
        same = torch.equal(y, product(h, 1))                            # the strips add up alike for any number of rows
        sd2.sd2_free(h)
        assert torch.cuda.mem_get_info()[0] == free0
        return "strips" if same else "cells"

    # (packing, the handle, its strips; then the dense weights on the device, the mask there, the cells)
    compress = lambda: sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4, sd2.SD2_DTYPE_F32)
    assert [served_by_strips(compress, k) for k in range(7)] == ["refused"] * 3 + ["strips"] * 3 + ["cells"]
    # (the dense weights on the host; the handle, its strips; the dense weights on the device, the cells)
    load = lambda: sd2.sd2_load_blob(blob, sd2.SD2_DTYPE_F32)
    assert [served_by_strips(load, k) for k in range(6)] == ["strips", "refused", "refused", "strips", "strips", "cells"]


def test_a_handle_tells_what_it_owns_and_what_a_call_reads():
    M, K = 1024, 2048
    W = synth.normal_bf16(41, (M, K), 0.02)
    mask = synth.bernoulli_mask(42, (M, K), 0.5)
    h = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4)
    one, many = sd2.sd2_spmm_query(h, 1), sd2.sd2_spmm_query(h, 40)
    assert (one["launches"], one["path"], one["streamed_bytes"]) == (1, sd2.SD2_PATH_STRIPS, h.compressed_bytes)
    assert (many["launches"], many["panel_rows"], many["path"]) == (2, 32, sd2.SD2_PATH_CELLS)
    assert 1.6 < many["streamed_bytes"] / (M * K) < 1.7                  # (three of four pairs have a word, at 50 %)
    assert one["device_bytes"] == many["device_bytes"] >= h.compressed_bytes + many["streamed_bytes"]
    sd2.sd2_debug_fail_allocations(5, 1)                                 # no memory for the cells
    try:
        bare = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4)
    finally:
        sd2.sd2_debug_fail_allocations(0, 0)
    facts = sd2.sd2_spmm_query(bare, 40)
    assert (facts["launches"], facts["panel_rows"], facts["path"]) == (10, 4, sd2.SD2_PATH_STRIPS)
    assert facts["device_bytes"] <= one["device_bytes"] - many["streamed_bytes"]
    asked = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4_STRIPS)        # the same, by choice
    assert sd2.sd2_spmm_query(asked, 40) == facts and asked.format == sd2.SD2_FORMAT_GAP4
    y = [torch.zeros((5, M), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    x = dev(synth.normal_bf16(43, (5, K), 1.0))
    sd2.sd2_spmm(bare, x, y[0])
    sd2.sd2_spmm(asked, x, y[1])
    sd2.sd2_stream_check()
    assert torch.equal(*y) and y[0].abs().max() > 0
    sd2.sd2_free(asked)
    bits, mma = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_BITMASK), sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4_MMA)
    assert [sd2.sd2_spmm_query(x, 65)[k] for x in (bits, mma) for k in ("launches", "path")] == [9, sd2.SD2_PATH_BITMASK, 2, sd2.SD2_PATH_MMA]
    for x in (h, bare, bits, mma):
        sd2.sd2_free(x)


def test_a_drafter_without_memory_for_its_cells_steps_through_the_strips():
    shape = synth.DrafterShape("small", 512, 128, 2048, 1)
    lin = synth.make_block(5, 0, shape, 0.5)
    hs = [sd2.sd2_compress(W, m, sd2.SD2_FORMAT_GAP4, sd2.SD2_DTYPE_F32 if i == 6 else sd2.SD2_DTYPE_BF16) for i, (W, m) in enumerate(lin)]
    x = dev(synth.make_activations(5, 0, 0, 8, shape.hidden))
    kinds = []
    for skip in range(24):
        sd2.sd2_debug_fail_allocations(skip, 1)
        try:
            d = sd2.sd2_drafter_create([hs], n_max=8)
        except sd2.Sd2Error as e:
            assert e.status == sd2.SD2_ERR_ALLOC
            kinds.append("refused")
            continue
        finally:
            sd2.sd2_debug_fail_allocations(0, 0)
        y = torch.full((8, shape.hidden), float("nan"), dtype=torch.float32, device="cuda")
        sd2.sd2_drafter_step(d, x, y)
        sd2.sd2_stream_check()
        t = _read_u16(sd2.sd2_drafter_buffers(d, 0)[6], 8 * shape.inter).reshape(8, -1)
        linear_close(y.double().cpu().numpy(), lin[6][0], lin[6][1], t, True)
        kinds.append("strips" if sd2.sd2_drafter_query(d, 8)["panel_rows"] == 4 else "cells")
        sd2.sd2_drafter_free(d)
    n = kinds.index("strips")
    assert kinds == ["refused"] * n + ["strips"] * 2 + ["cells"] * (22 - n)
    for h in hs:
        sd2.sd2_free(h)


@pytest.mark.parametrize("hidden,kv,inter,N", [(160, 48, 9600, 5),      # more gate tiles per cluster than wait for their up tiles at once
                                               (256, 64, 8192, 16)])    # the down projection in panels of its own
def test_block_over_cells(hidden, kv, inter, N):
    shape = synth.DrafterShape("tiny", hidden, kv, inter, 1)
    lin = synth.make_block(3, 0, shape, 0.5)
    hs = [sd2.sd2_compress(W, m, sd2.SD2_FORMAT_GAP4, sd2.SD2_DTYPE_F32 if i == 6 else sd2.SD2_DTYPE_BF16) for i, (W, m) in enumerate(lin)]
    x = synth.make_activations(3, 0, 0, N, hidden)
    ws = torch.full((sd2.sd2_block_workspace_bytes(hs, N) // 2,), float("nan"), dtype=torch.bfloat16, device="cuda")
    y = torch.full((N, hidden), float("nan"), dtype=torch.float32, device="cuda")
    for _ in range(2):                                                  # twice: the barrier words have to come back clean
        sd2.sd2_block_step(hs, dev(x), y, ws)
        sd2.sd2_stream_check()
    wsb = bits_of(ws)
    dims = [hidden, kv, kv, hidden, inter, inter, inter]
    q, k, v, hdn, g, u, t = [wsb[o // 2:o // 2 + N * d].reshape(N, d) for o, d in zip(sd2.sd2_block_workspace_layout(hs, N), dims)]
    for i, (inp, out) in enumerate([(x, q), (x, k), (x, v), (q, hdn), (hdn, g), (hdn, u)]):
        linear_close(values(out), lin[i][0], lin[i][1], inp, False)
    t_ref = values(np.array([oracle.f64_to_bf16_rne(float(z)) for z in oracle.silu_mul(g, u)], np.uint16)).reshape(N, -1)
    assert np.all(np.abs(values(t) - t_ref) <= 2.0 ** -6 * np.abs(t_ref))      # two ulp of bf16
    linear_close(y.double().cpu().numpy(), lin[6][0], lin[6][1], t, True)
    for h in hs:
        sd2.sd2_free(h)


@pytest.mark.parametrize("T,d", [(128, 64), (129, 64), (257, 128), (513, 8), (1100, 16)])     # clusters of one to eight
def test_attention_split_over_a_cluster(T, d):
    Hq, Hkv = 4, 2
    q = synth.normal_bf16(T, (1, Hq * d), 1.0)
    kc = synth.normal_bf16(T + 1, (1, T + 3, Hkv * d), 1.0)
    vc = synth.normal_bf16(T + 2, (1, T + 3, Hkv * d), 1.0)
    out = torch.full((1, Hq * d), float("nan"), dtype=torch.bfloat16, device="cuda")
    sd2.sd2_attention_decode(dev(q), dev(kc), dev(vc), out, Hq, Hkv, T)
    torch.cuda.synchronize()
    f64 = do.bf16_to_f64
    V = f64(vc[0, :T]).reshape(T, Hkv, d)
    ref = do.attention_decode(f64(q[0]).reshape(Hq, d), f64(kc[0, :T]).reshape(T, Hkv, d), V)
    # bf16 rounding, and fp32 arithmetic on weights that sum to one
    assert np.all(np.abs(f64(bits_of(out)).reshape(Hq, d) - ref) <= 2.0 ** -8 * np.abs(ref) + 2e-4 * np.abs(V).max())


@pytest.mark.parametrize("N,V,H", [(2, 1003, 72), (4, 5000, 264), (5, 50, 8), (1, 3, 8)])     # every width, shares of a few rows
def test_lm_head_widths(N, V, H):
    W = synth.normal_bf16(V, (V, H), 0.02)
    x = synth.normal_bf16(V + 1, (N, H), 1.0)
    logits = torch.full((N, V), float("nan"), dtype=torch.float32, device="cuda")
    toks = torch.full((N,), -1, dtype=torch.int32, device="cuda")
    sd2.sd2_lm_head(dev(x), dev(W), logits, toks)
    torch.cuda.synchronize()
    got = logits.double().cpu().numpy()
    linear_close(got, W, np.ones((V, H), np.uint8), x, True)
    assert [int(t) for t in toks] == [int(np.argmax(row)) for row in got]


@pytest.mark.parametrize("N", [1, 8])
def test_launches_that_overlap_still_run_in_order(N):
    # each product reads what the one before it wrote, and writes what the one before that read
    K = 1024
    W = synth.normal_bf16(7, (K, K), 0.045)
    h = sd2.sd2_compress(W, synth.bernoulli_mask(8, (K, K), 0.5))
    x = dev(synth.normal_bf16(9, (N, K), 1.0))

    def chain(wait):
        a, b = x.clone(), torch.zeros_like(x)
        for _ in range(40):
            sd2.sd2_spmm(h, a, b)
            if wait:
                torch.cuda.synchronize()
            a, b = b, a
        torch.cuda.synchronize()
        return a

    want = chain(True)
    assert torch.isfinite(want).all() and want.abs().max() > 0
    for _ in range(5):
        assert torch.equal(chain(False), want)
    sd2.sd2_free(h)


@pytest.mark.parametrize("fmt,N", [(sd2.SD2_FORMAT_GAP4, 1), (sd2.SD2_FORMAT_GAP4, 8), (sd2.SD2_FORMAT_GAP4_MMA, 16)])
def test_wait_budgets_do_not_count_the_kernel_before(fmt, N, monkeypatch):
    # weights that do not fit the ring, behind a launch of one CTA that leaves the other SMs free and takes longer than the
    # shortest budget: the launch streams weights ahead until its ring is full, and must then wait without a limit
    K_slow = 1 << 24
    slow = sd2.sd2_compress(np.full((1, K_slow), 0x3C00, np.uint16), np.ones((1, K_slow), np.uint8), sd2.SD2_FORMAT_BITMASK)
    xs = torch.ones((1, K_slow), dtype=torch.bfloat16, device="cuda")
    ys = torch.zeros((1, 1), dtype=torch.bfloat16, device="cuda")
    M, K = 8192, 4096
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    w = torch.empty((M, K), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=gen)
    h = sd2.sd2_compress(w, (torch.rand((M, K), device="cuda", generator=gen) < 0.5).to(torch.uint8), fmt)
    x = torch.empty((N, K), dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=gen)
    want, y = torch.zeros((N, M), dtype=torch.bfloat16, device="cuda"), torch.zeros((N, M), dtype=torch.bfloat16, device="cuda")
    sd2.sd2_spmm(h, x, want)
    sd2.sd2_spmm(slow, xs, ys)
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    start.record()
    sd2.sd2_spmm(slow, xs, ys)
    end.record()
    torch.cuda.synchronize()
    assert start.elapsed_time(end) > 3.0
    monkeypatch.setenv("SD2_WAIT_MS", "1")
    sd2.sd2_spmm(slow, xs, ys)
    sd2.sd2_spmm(h, x, y)
    sd2.sd2_stream_check()
    assert torch.isfinite(want).all() and torch.equal(y, want)                                       # (every format adds up in one order)
    for hh in (slow, h):
        sd2.sd2_free(hh)
