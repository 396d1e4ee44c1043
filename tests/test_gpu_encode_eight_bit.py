"""The throughput encoder's chain with 8-bit corrections: contiguous groups, 1024 codes and more, more than four tiles of 128 group
rows per SM (three from 1921 codes on), and codebooks without outliers and of codewords of like sizes.  Its error window is some fifty times that of the
half-precision chain, so these cases aim at it: planted pairs of codewords at gaps on both sides of the window, the
statistics taken in the same pass, and codebooks with outliers, which keep the half-precision chain at the same sizes."""
import numpy as np
import pytest
import torch

import paper_2410_15704_b200 as rvq
from helpers import assert_codes_match

pytestmark = pytest.mark.gpu


def kurtosis(cb):
    """Fourth moment of a stage's entries over the square of the second: 3 for a normal distribution."""
    e = cb.astype(np.float64).reshape(len(cb), -1)
    return (e ** 4).mean(axis=1) / (e ** 2).mean(axis=1) ** 2


def encode_both(x, cb, R, K):
    n = len(x)
    cfg = rvq.make_config(128, 32, rvq.CONTIGUOUS, R, K, 16, rvq.F32, 0)
    b, xd = rvq.alloc_buffers(cfg, n, cb), torch.from_numpy(x).cuda()
    exact = torch.empty_like(b.codes)
    rvq.rvq_encode(cfg, xd, n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    st = rvq.read_status(b.status)
    rvq.rvq_encode_exact(cfg, xd, n, 128, b.codebooks, b.prepared, exact, b.std, None)
    torch.cuda.synchronize()
    assert st["wait_timeouts"] == 0
    return cfg, b, xd, exact, st


@pytest.mark.parametrize("K,outliers", [(1024, False), (2048, False), (1024, True)])
def test_pairs_at_the_edge_of_the_window(K, outliers):
    """Every row has two codewords at nearly the same distance, relative gaps of 1e-3 ... 6e-2, either one ahead.  The
    window is some 9e-3 of the squared distance: half of the rows are compared exactly, the others certified right
    outside it, and all choices must be the float32 kernel's.  (outliers: some channels of the rows, not of the codewords.)"""
    g = np.random.default_rng(K)
    base = g.normal(size=(K // 8, 128))                                  # K / 2 group rows
    z = (base / base.std(axis=1, keepdims=True)).reshape(-1, 32)
    d = z[g.permutation(len(z))]
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    a = 0.2 * np.linalg.norm(z, axis=1, keepdims=True)
    gamma = np.exp(g.uniform(np.log(1e-3), np.log(6e-2), size=(len(z), 1)))
    pair = np.stack([z + a * d, z - a * (1.0 + 0.5 * gamma) * d], axis=1).reshape(K, 32)
    cb = pair[g.permutation(K)][None].astype(np.float32)
    assert kurtosis(cb).max() < 5.0
    x = np.repeat(base, 32768 // len(base), axis=0) * (1.0 + 1e-3 * g.normal(size=(32768, 128)))
    if outliers:
        x[::5, :3] *= 30.0
    x = x.astype(np.float32)
    cfg, b, _, exact, st = encode_both(x, cb, 1, K)
    assert torch.equal(b.codes, exact)
    codes = b.codes.view(torch.int16).cpu().numpy().view(np.uint16).reshape(len(x), 4, 1).astype(np.int32)
    assert_codes_match(x, codes, cb, rvq.CONTIGUOUS, sample=np.arange(0, len(x), 7))
    assert 0.2 < st["rescored_rows"] / (len(x) * 4) < 0.8 and st["exhaustive_rows"] < 0.1 * len(x)


@pytest.mark.parametrize("n,K", [(18945, 1024), (14219, 2048), (40000, 1030)])
def test_statistics_in_the_same_pass(n, K):
    """rvq_encode_stats where the chain has 8-bit corrections: the codes of rvq_encode, the counts and sums of rvq_ema_stats."""
    g = np.random.default_rng(n)
    R = 3
    x = g.normal(size=(n, 128)).astype(np.float32)
    cb = np.stack([g.normal(scale=0.8 ** r, size=(K, 32)) for r in range(R)]).astype(np.float32)
    assert kurtosis(cb).max() < 5.0
    cfg, b, xd, exact, _ = encode_both(x, cb, R, K)
    assert torch.equal(b.codes, exact)
    energy, fused_energy = torch.empty(R, device="cuda"), torch.empty(R, device="cuda")
    rvq.rvq_encode(cfg, xd, n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status, stage_energy=energy)
    count, total = torch.empty(R, K, device="cuda"), torch.empty(R, K, 32, device="cuda")
    rvq.rvq_ema_stats(cfg, xd, n, 128, b.codes, b.codebooks, count, total, b.workspace, b.workspace_bytes, b.status)
    f = rvq.alloc_buffers(cfg, n, cb)
    fused_count, fused_total = torch.full((R, K), -1.0, device="cuda"), torch.full((R, K, 32), 9.0, device="cuda")
    rvq.rvq_encode_stats(cfg, xd, n, 128, f.codebooks, f.prepared, f.codes, f.std, fused_count, fused_total, f.workspace, f.workspace_bytes,
                         f.status, stage_energy=fused_energy)
    torch.cuda.synchronize()
    assert torch.equal(f.codes, b.codes) and torch.equal(f.std, b.std) and torch.equal(fused_count, count)
    assert (torch.abs(fused_total - total) / count.clamp(min=1.0)[..., None]).max().item() <= 1e-4
    # (float32 additions of some 2e5 row energies each, warp by warp, in another order)
    assert torch.allclose(energy, fused_energy, rtol=1e-4)
    assert rvq.read_status(f.status)["wait_timeouts"] == 0


@pytest.mark.parametrize("n,K", [(18945, 1024), (14219, 2048)])
def test_codebooks_with_outliers(n, K):
    """Keys on contiguous groups: outlier channels, and codebooks that follow them."""
    g = np.random.default_rng(n)
    scale = 0.25 + np.abs(g.laplace(size=128))
    scale[g.permutation(128)[:8]] *= 20.0
    x = (g.normal(size=(n, 128)) * scale).astype(np.float32)
    unit = (scale / np.sqrt((scale ** 2).mean())).reshape(4, 32)
    cb = np.stack([g.normal(size=(K, 32)) * unit[g.integers(0, 4, size=K)] * 0.8 ** r for r in range(4)]).astype(np.float32)
    assert kurtosis(cb).min() > 8.0
    _, b, _, exact, st = encode_both(x, cb, 4, K)
    assert torch.equal(b.codes, exact)
    # (with 8-bit corrections 2-3 % of the rows and stages were compared exactly)
    assert st["rescored_rows"] + st["exhaustive_rows"] < 0.005 * n * 4 * 4


@pytest.mark.parametrize("n,K", [(18945, 1024), (14219, 2048)])
@pytest.mark.parametrize("kind,eight", [("group 10", True), ("group 1000", False), ("stages 1000", False)])
def test_codewords_of_different_sizes(n, K, kind, eight):
    """One of four groups smaller than the others, by 10 or 1000, in rows and codewords; half of the stages with outlier channels, the
    others even.  Rows far smaller than the largest codeword have many candidates under the 8-bit
    corrections (24 % and 22 % of the rows and stages, 20 times the time), so such codebooks keep the half-precision chain."""
    g = np.random.default_rng(n)
    R, what = 4, kind.split()
    scale = np.ones((R, 4, 32))
    if what[0] == "group":
        scale[:, 1] /= float(what[1])
    if what[0] == "stages":
        scale[:2, 0, :6] *= float(what[1])
    x = (g.normal(size=(n, 128)) * scale[0].reshape(-1)).astype(np.float32)
    scale /= np.sqrt((scale ** 2).mean(axis=(1, 2), keepdims=True))
    cb = np.stack([g.normal(size=(K, 32)) * scale[r, g.integers(0, 4, size=K)] * 0.8 ** r for r in range(R)]).astype(np.float32)
    assert np.sort(kurtosis(cb))[R // 2 - 1] < 6.0              # (even in at least half of the stages)
    _, b, _, exact, st = encode_both(x, cb, R, K)
    assert torch.equal(b.codes, exact)
    share = (st["rescored_rows"] + st["exhaustive_rows"]) / (n * 4 * R)
    assert 0.005 < share < 0.02 if eight else share < 0.01


@pytest.mark.parametrize("tiles,K,R,layout,statistics,factor", [(40, 2048, 3, 1, False, 20), (40, 1921, 2, 0, False, 20), (41, 2048, 2, 0, False, 1000),
                                                                (39, 2048, 2, 1, False, 200), (100, 1024, 2, 1, True, 20), (100, 1000, 2, 0, True, 1000)])
def test_long_calls_with_outliers(tiles, K, R, layout, statistics, factor):
    """Heavy-tailed keys and codebooks that follow them keep the half-precision chain however long the call is (with 8-bit
    corrections 45 % of the rows are compared at a factor of 1000, and the call takes 30 times as long): the codes are the
    float32 kernel's, and statistics taken in the pass are those of rvq_ema_stats."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = tiles * sms * 32 - (1 if tiles == 39 else 0)
    gen = torch.Generator(device="cuda").manual_seed(tiles + K)
    scale = 0.25 - torch.log(torch.rand(8, 128, generator=gen, device="cuda").clamp_min(1e-7))
    scale[:, ::16] *= factor
    x = (torch.randn((n + 7) // 8, 8, 128, generator=gen, device="cuda") * scale).view(-1, 128)[:n].contiguous()
    x[11] = 0.0
    unit = scale / scale.square().mean(dim=1, keepdim=True).sqrt()
    groups = (unit.view(8, 32, 4).transpose(1, 2) if layout else unit.view(8, 4, 32)).reshape(-1, 32)
    cb = torch.randn(R, K, 32, generator=gen, device="cuda") * groups[torch.randint(32, (R, K), generator=gen, device="cuda")]
    cb[1:] *= 0.8
    assert kurtosis(cb.cpu().numpy()).min() > 6.0
    cfg = rvq.make_config(128, 32, layout, R, K, 16, rvq.F32, 0)
    b = rvq.alloc_buffers(cfg, n, cb)
    exact = torch.empty_like(b.codes)
    got, want = [[torch.empty(R, K, device="cuda"), torch.empty(R, K, 32, device="cuda")] for _ in range(2)]
    if statistics:
        rvq.rvq_encode_stats(cfg, x, n, 128, b.codebooks, b.prepared, b.codes, b.std, *got, b.workspace, b.workspace_bytes, b.status)
        rvq.rvq_ema_stats(cfg, x, n, 128, b.codes, b.codebooks, *want, b.workspace, b.workspace_bytes, None)
        assert torch.equal(got[0], want[0])
        # (float32 sums of a bin's rows in another order, entries up to some 10 a row: the bound is a few ulps per row)
        assert ((got[1] - want[1]).abs() / want[0].clamp(min=1.0)[..., None]).max().item() <= 1e-4
    else:
        rvq.rvq_encode(cfg, x, n, 128, b.codebooks, b.prepared, b.codes, b.std, b.workspace, b.workspace_bytes, b.status)
    st = rvq.read_status(b.status)
    rvq.rvq_encode_exact(cfg, x, n, 128, b.codebooks, b.prepared, exact, b.std, None)
    torch.cuda.synchronize()
    assert torch.equal(b.codes, exact) and st["wait_timeouts"] == 0
    assert st["rescored_rows"] + st["exhaustive_rows"] < 0.005 * n * 4 * R


@pytest.mark.parametrize("n,K,R", [(4737, 2048, 2), (4737, 1921, 1), (9473, 1024, 2), (9473, 1030, 1), (9473, 2047, 2), (14209, 2048, 8)])
def test_packed_scores(n, K, R):
    """Codewords of like norms: scores in 16 bits, from two tiles per SM on (three with up to 1920 codes), also beside padding codewords.
    One codeword in four has a copy at 0 ... 1e-2 of its norm, which the window (some 2e-2 of a squared distance) cannot tell from
    it, and the rows' norms reach from 1e-3 to 2e4 times the codewords'."""
    g = np.random.default_rng(n + K)
    x = g.normal(size=(n, 128)).astype(np.float32)
    cb = np.stack([g.normal(scale=0.8 ** r, size=(K, 32)) for r in range(R)]).astype(np.float32)
    twin = g.permutation(K)[:2 * (K // 8)].reshape(2, -1)
    off = g.normal(size=(R, twin.shape[1], 32)) * np.exp(g.uniform(np.log(1e-6), np.log(2e-3), size=(1, twin.shape[1], 1)))
    cb[:, twin[1]] = cb[:, twin[0]] + (off * (g.random((1, twin.shape[1], 1)) < 0.9) * 0.8 ** np.arange(R)[:, None, None]).astype(np.float32)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert n * 4 > sms * 128 * (1 if K > 1920 else 2)
    _, b, _, exact, st = encode_both(x, cb, R, K)
    assert torch.equal(b.codes, exact) and st["rescored_rows"] > 0.1 * n * 4 * R
    # (the first group of every third row carries next to all of its energy, or next to none)
    x[::3, :32] *= np.exp(g.uniform(np.log(1e-3), np.log(1e3), size=(len(x[::3]), 1))).astype(np.float32)
    for scale in (1.0, 1e-3, 20.0, 2e-4):
        _, b, _, exact, _ = encode_both(x, (cb * scale).astype(np.float32), R, K)
        assert torch.equal(b.codes, exact)
    # (exact ties: the lowest index)
    cb[:, twin[1]] = cb[:, twin[0]]
    _, b, _, exact, _ = encode_both(x, cb, R, K)
    assert torch.equal(b.codes, exact)
