"""The encoders that split a row's codebook over several CTAs (few head vectors), at the sizes where a
dispatch or a split can go wrong: codes, deviations and stage energies against the all-float32 kernel."""
import numpy as np
import pytest
import torch

import oracle
import paper_2410_15704_b200 as rvq
from helpers import DT, RECON_TOL, assert_codes_match, codes_to_numpy
import test_gpu_learning

pytestmark = pytest.mark.gpu


def batch(n, dim, K, R, dtype, seed):
    g = np.random.default_rng(seed)
    scale = np.where(g.random(dim) < 0.06, 20.0, 1.0)
    x = torch.from_numpy((g.normal(size=(n, dim)) * scale).astype(np.float32)).to(rvq.TORCH_DTYPE[DT[dtype]])
    if n % 2 == 1 and n > 3:
        x[2] = 0.0                                          # degenerate
    cb = np.stack([g.normal(scale=0.8 ** r, size=(K, 32)) for r in range(R)]).astype(np.float32)
    if K > 40:
        cb[0, 40] = cb[0, 3]                                # duplicates: the lower index wins
    return x, cb


def check(n, dim, K, R, layout, bits, dtype, seed, stride=None):
    x, cb = batch(n, dim, K, R, dtype, seed)
    cfg = rvq.make_config(dim, 32, layout, R, K, (K - 1).bit_length() if bits == "packed" else 16, DT[dtype], seed % 2)
    stride = stride or dim
    xd = torch.zeros(n, stride, dtype=x.dtype, device="cuda")
    xd[:, :dim] = x.cuda()
    b, e = rvq.alloc_buffers(cfg, n, cb), rvq.alloc_buffers(cfg, n, cb)
    energy, energy_e = torch.full((R,), 7.0, device="cuda"), torch.empty(R, device="cuda")
    for out in (None, energy):                              # with and without the stage energies
        b.codes.fill_(0xAA)
        rvq.rvq_encode(cfg, xd, n, stride, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes,
                       b.status, stage_energy=out)
        rvq.rvq_encode_exact(cfg, xd, n, stride, e.codebooks, e.prepared, e.codes, e.std, e.status, stage_energy=energy_e)
        torch.cuda.synchronize()
        assert torch.equal(b.codes, e.codes) and torch.equal(b.std, e.std)
    assert torch.allclose(energy, energy_e, rtol=1e-4)
    st, ste = rvq.read_status(b.status), rvq.read_status(e.status)
    assert st["wait_timeouts"] == 0 and st["degenerate_vectors"] == ste["degenerate_vectors"]


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 9, 17, 31, 32, 33, 63, 64, 65, 127, 129, 257, 600, 1111, 2049])
@pytest.mark.parametrize("K,R,layout,bits,dtype", [(2048, 8, 1, "packed", "bf16"), (1024, 8, 0, 16, "f32"),
                                                   (1000, 5, 1, "packed", "f16"), (256, 8, 0, 16, "f32"), (77, 3, 0, "packed", "bf16")])
def test_few_vectors(n, K, R, layout, bits, dtype):
    check(n, 128, K, R, layout, bits, dtype, n + K)


@pytest.mark.parametrize("n", [1, 3, 5, 8, 15, 16, 17, 33])
@pytest.mark.parametrize("dim,K,R,layout,bits,dtype", [(128, 2048, 8, 1, "packed", "bf16"), (128, 1300, 8, 0, 16, "f32"), (256, 600, 4, 0, "packed", "f16"),
                                                       (128, 2, 8, 1, "packed", "f32"), (128, 16, 2, 0, "packed", "f32"), (64, 1025, 8, 1, 16, "bf16"),
                                                       (512, 1024, 8, 1, "packed", "bf16"), (1024, 512, 8, 0, "packed", "f32")])
def test_groups_of_a_vector_shared_out(n, dim, K, R, layout, bits, dtype):
    """Clusters that take one or two of a head vector's groups each, in as many as run at a time and beyond, and write the
    bytes of their rows' codes: one to eleven bits a code, one to sixteen blocks of codewords."""
    check(n, dim, K, R, layout, bits, dtype, n + K, stride=dim + 16)


@pytest.mark.parametrize("n,dim,K", [(5, 256, 2048), (70, 256, 1024), (301, 64, 512), (9, 32, 2048), (40, 96, 300), (3, 512, 129),
                                     (13000, 128, 512), (150, 128, 5000), (4, 1024, 2049)])
def test_other_head_sizes_and_row_strides(n, dim, K):
    check(n, dim, K, 8 if K != 129 else 9, 1, "packed", "bf16", n, stride=dim + 16)


@pytest.mark.parametrize("tiles", [1, 19, 37, 74, 148])
@pytest.mark.parametrize("K", [100, 140, 256, 384, 400, 520, 770, 1024, 1400, 2048, 5000])
def test_chunks_over_accumulators_and_ctas(tiles, K):
    """Up to three chunks: one tile per CTA, an accumulator per chunk.  More: tiles split over one to eight CTAs of one to forty chunks each: chains that go out together and one by one, groups
    without a chunk, slots and accumulators that come round; equal codewords in different chunks, groups and CTAs."""
    n = 32 * tiles - tiles % 3
    x, cb = batch(n, 128, K, 5, "bf16", tiles + K)
    cb[:, min(130, K - 2)], cb[:, K - 1], cb[:, K // 2] = cb[:, 2], cb[:, 5], cb[:, 9]
    cfg = rvq.make_config(128, 32, 1, 5, K, 16, rvq.BF16, 0)
    b = rvq.alloc_buffers(cfg, n, cb)
    exact = torch.empty_like(b.codes)
    rvq.rvq_encode(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    rvq.rvq_encode_exact(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, exact, b.std, b.status)
    torch.cuda.synchronize()
    assert torch.equal(b.codes, exact) and rvq.read_status(b.status)["wait_timeouts"] == 0


@pytest.mark.parametrize("n,K,layout", [(5000, 1024, 1), (19000, 1024, 0), (900, 1024, 1), (500, 384, 0), (40, 2048, 1)])
@pytest.mark.parametrize("copies", [2, 3, 8])
def test_rows_with_many_candidates(n, K, layout, copies):
    """Every codeword there several times, some copies moved a little: each row has candidates in two, three or all
    chunks, and the rows of a warp are compared four at a time; the lowest index wins among equals."""
    x, cb = batch(n, 128, K, 4, "bf16", n + copies)
    step = K // copies
    for c in range(1, copies):
        cb[:, c * step:(c + 1) * step] = cb[:, :step] * (1.0 + 1e-6 * (c % 2))
    cfg = rvq.make_config(128, 32, layout, 4, K, 16, rvq.BF16, 0)
    b = rvq.alloc_buffers(cfg, n, cb)
    exact = torch.empty_like(b.codes)
    rvq.rvq_encode(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    rvq.rvq_encode_exact(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, exact, b.std, b.status)
    torch.cuda.synchronize()
    assert torch.equal(b.codes, exact) and rvq.read_status(b.status)["wait_timeouts"] == 0


@pytest.mark.parametrize("tiles", [149, 296, 400, 592, 740, 1030, 1184])
@pytest.mark.parametrize("K,R,layout", [(100, 3, 1), (256, 8, 0), (600, 1, 0), (1024, 4, 1), (1500, 2, 0)])
def test_rounds_of_two_and_three_tiles(tiles, K, R, layout):
    """One to eight tiles per SM: rounds of one, two and three tiles and one kind after the other, among them calls in which some
    CTAs have a tile more than others; codebooks of one to twelve chunks; a last tile that is not full."""
    n = 32 * tiles - 5
    x, cb = batch(n, 128, K, R, "bf16", tiles + K)
    cfg = rvq.make_config(128, 32, layout, R, K, 16, rvq.BF16, 0)
    b = rvq.alloc_buffers(cfg, n, cb)
    exact = torch.empty_like(b.codes)
    for _ in range(2):
        b.codes.fill_(0xAA)
        rvq.rvq_encode(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
        rvq.rvq_encode_exact(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, exact, b.std, b.status)
        torch.cuda.synchronize()
        assert torch.equal(b.codes, exact) and rvq.read_status(b.status)["wait_timeouts"] == 0


@pytest.mark.parametrize("n,dim,K,R,layout,dtype", [(14209, 128, 256, 2, 1, "bf16"), (20003, 128, 1024, 3, 1, "f32"), (19001, 128, 1024, 2, 0, "f16"),
                                                    (7150, 256, 600, 2, 0, "f32"), (60001, 32, 300, 2, 0, "bf16"), (1801, 1024, 400, 2, 1, "bf16")])
@pytest.mark.parametrize("gap", [0, 16, 1000])
def test_rows_of_the_rounds_to_come(n, dim, K, R, layout, dtype, gap):
    """More than three tiles per SM, so that every CTA, or some, ask for the rows of a second round while the first runs: as one run where
    the rows lie without gaps, vector by vector where they do not, up to a last round that ends inside a tile.  Rows with gaps are the
    last thing in their allocation."""
    x, cb = batch(n, dim, K, R, dtype, n + gap)
    cfg = rvq.make_config(dim, 32, layout, R, K, 16, DT[dtype], 0)
    stride = dim + gap
    xd = torch.full(((n - 1) * stride + dim,), float("nan"), dtype=x.dtype, device="cuda").as_strided((n, dim), (stride, 1))
    xd.copy_(x)
    b, e = rvq.alloc_buffers(cfg, n, cb), rvq.alloc_buffers(cfg, n, cb)
    rvq.rvq_encode(cfg, xd, n, stride, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    rvq.rvq_encode_exact(cfg, x.cuda(), n, dim, e.codebooks, e.prepared, e.codes, e.std, e.status)
    torch.cuda.synchronize()
    assert torch.equal(b.codes, e.codes) and torch.equal(b.std, e.std) and rvq.read_status(b.status)["wait_timeouts"] == 0


def test_against_the_oracle():
    x, cb = batch(24, 128, 1024, 8, "f32", 5)
    cfg = rvq.make_config(128, 32, 0, 8, 1024, 16, rvq.F32, 0)
    b = rvq.alloc_buffers(cfg, 24, cb)
    rvq.rvq_encode(cfg, x.cuda(), 24, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    codes = b.codes.view(torch.int16).cpu().numpy().view(np.uint16).reshape(24, 4, 8).astype(np.int32)
    assert_codes_match(x.numpy(), codes, cb, 0)


@pytest.mark.parametrize("n,K,R,scale", [(18945, 1024, 8, 1.0), (14219, 2048, 4, 1.0), (18960, 1030, 2, 1e-3), (19000, 1024, 2, 3e4)])
def test_eight_bit_corrections(n, K, R, scale):
    """Contiguous groups, eight or more chunks, more than four tiles per SM (three with 2048 codes): ordinary codebooks, and ones whose
    stages' scales lie far apart (rows beyond the 8-bit range take the full scan)."""
    x, cb = batch(n, 128, K, R, "f32", n)
    cb[0, ::7] *= 8.0
    cb[-1] *= scale
    cfg = rvq.make_config(128, 32, 0, R, K, 16, rvq.F32, 0)
    b = rvq.alloc_buffers(cfg, n, cb)
    exact = torch.empty_like(b.codes)
    rvq.rvq_encode(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    rvq.rvq_encode_exact(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, exact, b.std, b.status)
    torch.cuda.synchronize()
    assert torch.equal(b.codes, exact) and rvq.read_status(b.status)["wait_timeouts"] == 0


@pytest.mark.parametrize("n,dim,K,R,layout", [(1, 128, 1024, 8, 0), (33, 128, 512, 4, 1), (2055, 128, 1000, 8, 1), (1025, 256, 2048, 6, 0), (5003, 256, 512, 8, 1),
                                              (4737, 128, 1024, 2, 0)])
def test_statistics_of_few_tiles(n, dim, K, R, layout):
    """Batches whose statistics are taken by the separate pass, with four groups and eight (the last one: fused), against float64."""
    x, cb = batch(n, dim, K, R, "f32", n)
    x[2 % n] = x[0]                                         # (no degenerate row)
    cfg = rvq.make_config(dim, 32, layout, R, K, 16, rvq.F32, 0)
    b, G, xd = rvq.alloc_buffers(cfg, n, cb), dim // 32, x.cuda()
    count, total = torch.empty(R, K, device="cuda"), torch.empty(R, K, 32, device="cuda")
    rvq.rvq_encode_stats(cfg, xd, n, dim, b.codebooks, b.prepared, b.codes, b.std, count, total, b.workspace, b.workspace_bytes, b.status)
    codes = (b.codes.view(torch.int16).view(n, -1)[:, :G * R].reshape(n * G, R).long() & 0xFFFF)
    z = xd.double() / xd.double().std(dim=1, unbiased=False, keepdim=True)
    z = (z.view(n, 32, G).transpose(1, 2) if layout else z.view(n, G, 32)).reshape(n * G, 32)
    for r in range(R):
        assert torch.equal(count[r].long(), torch.bincount(codes[:, r], minlength=K))
        want = torch.zeros(K, 32, dtype=torch.float64, device="cuda").index_add_(0, codes[:, r], z)
        assert (total[r].double() - want).abs().max() <= 1e-5 * max(1.0, want.abs().max().item())
        z = z - b.codebooks.view(R, K, 32)[r][codes[:, r]].double()


@pytest.mark.parametrize("n,dim,K,R,layout", [(4096, 32, 512, 8, 0), (4097, 32, 512, 8, 0), (1200, 64, 300, 8, 1), (1201, 64, 300, 8, 1),
                                              (256, 512, 1024, 8, 1), (257, 512, 1024, 8, 1), (1024, 128, 1024, 12, 0), (1025, 128, 1024, 12, 0),
                                              (8, 1024, 512, 8, 1), (8, 1024, 1023, 4, 0), (700, 128, 6000, 8, 0), (2048, 128, 512, 4, 1), (2049, 128, 512, 4, 1),
                                              (1100, 256, 550, 8, 0), (1101, 256, 550, 8, 0)])
def test_statistics_by_the_other_passes(n, dim, K, R, layout):
    """The same on both sides of the lines between fused statistics and a pass of their own, for head vectors of one, two,
    four, eight, sixteen and thirty-two groups, more than eight stages, and more codes than a histogram in shared memory holds."""
    test_statistics_of_few_tiles(n, dim, K, R, layout)


@pytest.mark.parametrize("n,dim,K,R,layout", [(4737, 128, 1024, 4, 1), (18945, 128, 1024, 3, 0), (8000, 64, 300, 3, 0), (20000, 128, 256, 1, 0), (600, 128, 1024, 4, 0)])
def test_statistics_of_degenerate_vectors(n, dim, K, R, layout):
    """Vectors of zero or non-finite deviation have codes 0 and count for them, and their stage inputs are what those codes
    leave of zero: statistics taken in the encoder's pass (all cases but the last) are those of rvq_ema_stats, and the oracle's."""
    x, cb = batch(n, dim, K, R, "f32", 2 * n)
    x[::97] = 0.0
    x[5, 3], x[n - 1, 0] = float("nan"), float("inf")
    cfg = rvq.make_config(dim, 32, layout, R, K, 16, rvq.F32, 0)
    b, xd = rvq.alloc_buffers(cfg, n, cb), x.cuda()
    got, want = [[torch.empty(R, K, device="cuda"), torch.empty(R, K, 32, device="cuda")] for _ in range(2)]
    rvq.rvq_encode_stats(cfg, xd, n, dim, b.codebooks, b.prepared, b.codes, b.std, *got, b.workspace, b.workspace_bytes, b.status)
    rvq.rvq_ema_stats(cfg, xd, n, dim, b.codes, b.codebooks, *want, b.workspace, b.workspace_bytes, b.status)
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0])
    # (float32 sums of up to a bin's count of rows in another order, and a codeword subtracted and added back)
    scale = want[0].clamp(min=1.0)[..., None]
    assert ((got[1] - want[1]).abs() / scale).max().item() <= 1e-4
    codes = codes_to_numpy(cfg, b.codes, n)
    assert not codes[::97].any()
    count, total = oracle.ema_stats(x.numpy(), codes, cb, layout)
    assert np.array_equal(got[0].cpu().numpy(), count)
    assert np.max(np.abs(got[1].cpu().numpy() - total) / scale.cpu().numpy()) <= 1e-4


@pytest.mark.parametrize("n,K", [(5, 1024), (601, 1024), (4001, 256), (601, 256)])
def test_stage_energy_leaves_degenerate_vectors_out(n, K):
    """In every encoder: the energies of a batch with vectors of zero and non-finite deviation are those of the others."""
    x, cb = batch(n, 128, K, 3, "f32", 2 * n)
    x[::4] = 0.0
    x[1, 3], x[n - 2, 0] = float("nan"), float("inf")
    keep = torch.isfinite(x).all(dim=1) & (x != 0).any(dim=1)
    cfg = rvq.make_config(128, 32, 0, 3, K, 16, rvq.F32, 0)
    z = oracle.encode(x[keep].numpy(), cb, 32, 0, want_residual=True)
    last = float((z["residual"] ** 2).sum())
    for exact in (False, True):
        b, energy = rvq.alloc_buffers(cfg, n, cb), torch.empty(3, device="cuda")
        if exact:
            rvq.rvq_encode_exact(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, b.codes, b.std, b.status, stage_energy=energy)
        else:
            rvq.rvq_encode(cfg, x.cuda(), n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status,
                           stage_energy=energy)
        torch.cuda.synchronize()
        assert abs(energy[-1].item() - last) <= 1e-4 * last       # (float32 additions of row energies, in any order)


@pytest.mark.parametrize("seed", range(4))
def test_quotients_of_the_encoder_are_those_of_a_division(seed):
    """The throughput encoder divides a row by its deviation with corrected reciprocals, or one by one where a value is
    outside a wide range of exponents.  Every row has a codeword of its own here, so that the sum of a bin is one row's
    scaled values, bit for bit; rvq_ema_stats with 16 groups divides.  Half of the vectors keep to the ordinary range, the
    others hold elements far below and above it, deviations beyond it on both sides, and zeros."""
    g = np.random.default_rng(seed)
    dim, K, live, n = 512, 4096, 256, 1300
    x = g.normal(size=(live, dim))
    x[:128] *= 2.0 ** g.integers(-38, 39, size=(128, 1))
    wild = x[128:]
    wild[:32] *= 2.0 ** -g.integers(62, 140, size=(32, dim)) ** (g.random((32, dim)) < 0.1)
    wild[32:64] *= 2.0 ** g.integers(41, 60, size=(32, 1))
    wild[64:96] *= 2.0 ** -g.integers(41, 55, size=(32, 1))
    wild[96:][g.random((32, dim)) < 0.2] = 0.0
    wild[112:, 0] *= 2.0 ** 10
    x = np.concatenate([x, np.zeros((n - live, dim))]).astype(np.float32)
    z = x[:live].astype(np.float64)
    z = (z / z.std(axis=1, keepdims=True)).reshape(-1, 32)
    cb = z[g.permutation(K)][None].astype(np.float32)
    cfg = rvq.make_config(dim, 32, 0, 1, K, 16, rvq.F32, 0)
    b, xd = rvq.alloc_buffers(cfg, n, cb), torch.from_numpy(x).cuda()
    got, want = [[torch.empty(1, K, device="cuda"), torch.empty(1, K, 32, device="cuda")] for _ in range(2)]
    rvq.rvq_encode_stats(cfg, xd, n, dim, b.codebooks, b.prepared, b.codes, b.std, *got, b.workspace, b.workspace_bytes, b.status)
    rvq.rvq_ema_stats(cfg, xd, n, dim, b.codes, b.codebooks, *want, b.workspace, b.workspace_bytes, b.status)
    torch.cuda.synchronize()
    assert len(np.unique(codes_to_numpy(cfg, b.codes, n)[:live])) == K
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("dim,gd,K,R", [(32, 32, 300, 3), (32, 32, 1024, 1), (32, 32, 600, 9), (96, 32, 129, 5), (24, 8, 50, 3), (64, 64, 70, 1)])
@pytest.mark.parametrize("n", [1, 2, 700])
def test_odd_numbers_of_16_bit_codes(dim, gd, K, R, n):
    """uint16 codes are [n][G][R] without gaps also where a vector has an odd number of them, for what writes and what reads them."""
    g = np.random.default_rng(dim + K + R + n)
    x = g.normal(size=(n, dim)).astype(np.float32)
    cb = np.stack([g.normal(scale=0.8 ** r, size=(K, gd)) for r in range(R)]).astype(np.float32)
    cfg = rvq.make_config(dim, gd, 1, R, K, 16, rvq.F32, 0)
    assert rvq.rvq_code_bytes(cfg) == dim // gd * R * 2
    b, xd = rvq.alloc_buffers(cfg, n, cb), torch.from_numpy(x).cuda()
    out, rotated = torch.empty_like(xd), torch.empty_like(xd)
    count, total = torch.empty(R, K, device="cuda"), torch.empty(R, K, gd, device="cuda")
    table, pos = torch.empty(1, dim // 2, 2, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    rvq.rvq_rope_table(dim, 10000.0, 1, table)                             # position 0: nothing is rotated
    rvq.rvq_encode(cfg, xd, n, dim, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    rvq.rvq_decode(cfg, b.codes, b.std, n, b.codebooks, b.prepared, out, dim, b.status)
    rvq.rvq_decode_rope(cfg, b.codes, b.std, n, b.codebooks, b.prepared, pos, 1, table, 1, rvq.ROPE_HALVES, rotated, dim, b.status)
    rvq.rvq_ema_stats(cfg, xd, n, dim, b.codes, b.codebooks, count, total, b.workspace, b.workspace_bytes, b.status)
    torch.cuda.synchronize()
    codes = codes_to_numpy(cfg, b.codes, n)
    assert_codes_match(x, codes, cb, 1)
    want = oracle.decode(codes, b.std.cpu().numpy().view(np.uint16)[:n], cb, dim, 1)
    assert np.abs(out.cpu().numpy() - want).max() <= RECON_TOL and np.abs(rotated.cpu().numpy() - want).max() <= RECON_TOL
    want_count, want_total = oracle.ema_stats(x, codes, cb, 1)
    assert np.array_equal(count.cpu().numpy(), want_count)
    assert np.max(np.abs(total.cpu().numpy() - want_total) / np.maximum(1.0, want_count)[..., None]) <= 1e-4
    assert rvq.read_status(b.status)["bad_codes"] == 0


@pytest.mark.parametrize("layout", [0, 1])
def test_kmeans_of_one_group(layout):
    test_gpu_learning.test_kmeans_init_on_separated_clusters(layout, 1)


@pytest.mark.parametrize("K,gd", [(2, 8), (33, 64), (1000, 32), (2048, 32)])
def test_update_of_buffers_that_are_not_aligned(K, gd):
    """rvq_ema_apply on buffers that start 4 bytes past a 16-byte boundary equals that on aligned ones."""
    g = torch.Generator(device="cuda").manual_seed(K)
    cfg = rvq.make_config(gd * 4, gd, 0, 3, K, 16, rvq.F32, 0)
    count, total = torch.rand(3, K, device="cuda", generator=g), torch.randn(3, K, gd, device="cuda", generator=g)
    state = [torch.rand(3, K, device="cuda", generator=g) + 0.1, torch.randn(3, K, gd, device="cuda", generator=g), torch.zeros(3, K, gd, device="cuda")]
    want = [t.clone() for t in state]
    rvq.rvq_ema_apply(cfg, count, total, want[2], want[0], want[1], 0.9, 1e-5)
    shifted = [torch.empty(t.numel() + 1, device="cuda")[1:].view(t.shape).copy_(t) for t in state + [total]]
    rvq.rvq_ema_apply(cfg, count, shifted[3], shifted[2], shifted[0], shifted[1], 0.9, 1e-5)
    for a, b in zip(shifted, want):
        assert torch.equal(a, b)
