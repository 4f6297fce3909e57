"""mma_kernel at the sizes where it changes: edges of blocks and panels, shares of a panel's columns, waves of clusters.

Products are exact; a team's sum takes K / 64 steps of the tensor core at most, each truncated to within 2^-22 of S = sum |w x|, and
the sums of four teams and eight shares meet in fp32: |y - ref| <= (K / 64 + 12) * 2^-22 S.  bf16 outputs add 2^-8 |y|.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle
from paper_2504_08838_b200 import binding as sd2
from paper_2504_08838_b200 import synth
from tests.test_gpu_cells import bits_of, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,density,shift", [
    (1, 8, 1, 1.0, 0), (128, 64, 16, 0.5, 0), (129, 65, 17, 0.5, 0),          # one block; a row, a column more
    (128, 512, 48, 0.5, 0), (31, 520, 33, 0.5, 0),                            # a block for every share of eight, one share with two
    (100, 4100, 64, 0.5, 0), (100, 4101, 5, 0.5, 0), (77, 1000, 20, 0.5, 1),  # whole rounds and a rest; rows that are not aligned
    (640, 2048, 24, 0.02, 0), (640, 2048, 64, 1.0, 0), (640, 2048, 32, 0.0, 0),   # small copies, the largest blocks, nothing kept
    (3072, 1000, 16, 0.3, 0), (19201, 72, 3, 0.5, 0), (9600, 200, 40, 0.5, 3),    # five shares; more panels than SMs; two shares
])
def test_panels(M, K, N, density, shift):
    W = synth.normal_bf16(M + K, (M, K), 0.02)
    mask = synth.bernoulli_mask(M + K + 1, (M, K), density) if 0.0 < density < 1.0 else np.full((M, K), int(density), np.uint8)
    x = synth.normal_bf16(M + K + 2, (N, K), 1.0)
    f32 = N % 2 == 0
    h = sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4_MMA, sd2.SD2_DTYPE_F32 if f32 else sd2.SD2_DTYPE_BF16)
    assert np.array_equal(sd2.sd2_decompress(h), oracle.roundtrip_ref(W, mask))
    store = torch.zeros(N * K + shift, dtype=torch.bfloat16, device="cuda")
    store[shift:] = dev(x).view(-1)
    guard = 40
    buf = torch.full((N * M + 2 * guard,), float("nan"), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    y = buf[guard:guard + N * M].view(N, M)
    sd2.sd2_spmm(h, store[shift:].view(N, K), y)
    sd2.sd2_stream_check()
    first = y.clone()
    out = buf.float().cpu().numpy().astype(np.float64)
    assert np.isnan(out[:guard]).all() and np.isnan(out[-guard:]).all() and not np.isnan(out[guard:-guard]).any()
    ref, S = oracle.masked_linear(W, mask, x)
    tol = (K / 64 + 12) * 2.0 ** -22 * S
    assert np.all(np.abs(out[guard:-guard].reshape(N, M) - ref) <= tol + (0.0 if f32 else 2.0 ** -8 * (np.abs(ref) + tol)))
    # the same sums in every call, alone and among others, in two streams at once
    streams = [torch.cuda.Stream() for _ in range(2)]
    ys = [torch.zeros_like(first) for _ in streams]
    torch.cuda.synchronize()
    for _ in range(3):
        for s, o in zip(streams, ys):
            sd2.sd2_spmm(h, store[shift:].view(N, K), o, stream=s.cuda_stream)
    one = torch.zeros_like(first[:1])
    sd2.sd2_spmm(h, store[shift:].view(N, K)[N - 1:], one)
    torch.cuda.synchronize()
    assert all(torch.equal(o, first) for o in ys) and torch.equal(one, first[N - 1:])
    sd2.sd2_free(h)


@pytest.mark.parametrize("M,K,density", [(130, 264, 0.5), (257, 129, 1.0), (300, 1000, 0.02), (64, 4099, 0.1), (1, 1, 1.0), (129, 65, 0.0)])
def test_the_facts_of_a_panel_handle_are_those_of_its_blob(M, K, density):
    W = synth.normal_bf16(M + K, (M, K), 0.02)
    mask = synth.bernoulli_mask(M + K + 1, (M, K), density) if 0.0 < density < 1.0 else np.full((M, K), int(density), np.uint8)
    for m in (mask, None):
        want = sd2.sd2_unpack_host(sd2.sd2_pack_host(W, m, sd2.SD2_FORMAT_GAP4_MMA), want_dense=False)[1]
        h = sd2.sd2_compress(W, m, sd2.SD2_FORMAT_GAP4_MMA)
        assert {k: v for k, v in sd2.sd2_info(h).items() if k in want} == want
        sd2.sd2_free(h)


def test_panel_handles_are_made_in_little_memory():
    # 8200 rows are made in five parts, the last of eight rows, in the 48 MiB beside the handle that a part of the weights and its mask
    # take (all of them take 201 MB)
    M = K = 8192
    M += 8
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    w = torch.empty((M, K), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=gen)
    w.masked_fill_(w == 0, 0.02)                                          # (a loaded handle has no words for kept zeros)
    m = (torch.rand((M, K), device="cuda", generator=gen) < 0.25).to(torch.uint8)
    x = torch.empty((16, K), dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=gen)
    h = sd2.sd2_compress(w, m, sd2.SD2_FORMAT_GAP4_MMA)                   # in place: in one part
    want = torch.zeros((16, M), dtype=torch.bfloat16, device="cuda")
    sd2.sd2_spmm(h, x, want)
    sd2.sd2_stream_check()
    need = sd2.sd2_spmm_query(h, 16)["device_bytes"]
    W, mask = bits_of(w), m.cpu().numpy()
    dense = sd2.sd2_decompress(h)
    assert np.array_equal(dense, oracle.roundtrip_ref(W, mask))
    sd2.sd2_free(h)
    blob = sd2.sd2_pack_host(W, mask, sd2.SD2_FORMAT_GAP4_MMA)
    y = torch.zeros_like(want)
    del w, m
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - need - (72 << 20), dtype=torch.uint8, device="cuda")
    assert need + (48 << 20) < torch.cuda.mem_get_info()[0] < need + (96 << 20)
    for make in (lambda: sd2.sd2_load_blob(blob), lambda: sd2.sd2_compress(W, mask, sd2.SD2_FORMAT_GAP4_MMA)):
        h = make()
        assert sd2.sd2_spmm_query(h, 16)["device_bytes"] == need and np.array_equal(sd2.sd2_decompress(h), dense)
        sd2.sd2_spmm(h, x, y.zero_())
        sd2.sd2_stream_check()
        assert torch.equal(y, want)
        sd2.sd2_free(h)
    del hog
    torch.cuda.empty_cache()


def test_a_loaded_panel_handle_decompresses_bit_for_bit():
    M, K = 130, 200
    W = synth.normal_bf16(51, (M, K), 0.02)
    mask = synth.bernoulli_mask(52, (M, K), 0.5)
    mask[0, :5] = 1
    W[0, :5] = (0x8000, 0x0000, 0x7FC1, 0xFF80, 0x0001)                  # a kept -0 and +0, NaN, -infinity, the smallest
    h = sd2.sd2_load_blob(sd2.sd2_pack_host(W, mask, sd2.SD2_FORMAT_GAP4_MMA))
    assert np.array_equal(sd2.sd2_decompress(h), oracle.roundtrip_ref(W, mask))
    x = np.zeros((1, K), np.uint16)
    x[0, 4] = 0x3F80
    y = torch.zeros((1, M), dtype=torch.bfloat16, device="cuda")
    sd2.sd2_spmm(h, dev(x), y)
    sd2.sd2_stream_check()
    assert np.array_equal(bits_of(y)[0, 1:], oracle.roundtrip_ref(W, mask)[1:, 4])
    sd2.sd2_free(h)
