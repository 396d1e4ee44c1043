"""The decoders that keep tables in shared memory, at the sizes and shapes for which they are chosen (decode_direct_wanted,
csrc/decode_direct.cu): four groups from 28673 vectors, rotated from 131073, eight groups from 32769, and head vectors of
one or two groups.  Few vectors of four groups and more take their codewords from L2 instead, so smaller batches do not
come here.  Reconstructions against the oracle; that the tables were used is seen by a few elements that round otherwise
than the float32 sums in stage order, which a small batch of the same vectors gives."""
import numpy as np
import pytest
import torch

import oracle
import paper_2410_15704_b200 as rvq
import rvq_synth
from helpers import DT, HALF_ULP, RECON_TOL, assert_recon_match, codes_to_device

pytestmark = pytest.mark.gpu

HEADS, BASE, POSITIONS = 8, 500000.0, 5000
C, S = rvq_synth.CONTIGUOUS, rvq_synth.STRIDED


def make(n, dim, K, R, std_scale, outlier_every, seed):
    g = np.random.default_rng(seed)
    codes = g.integers(0, K, size=(n, dim // 32, R)).astype(np.int32)
    std = std_scale * (np.abs(1.0 + 0.25 * g.normal(size=n)) + 0.05)
    if outlier_every:
        std[::outlier_every] *= 50.0                        # single rows beyond the chosen table's reach
    cb = np.stack([g.normal(scale=0.5 * 0.75 ** r, size=(K, 32)) for r in range(R)]).astype(np.float32)
    return codes, std.astype(np.float16).view(np.uint16), cb, g.integers(0, POSITIONS, size=-(-n // HEADS)).astype(np.int32)


def run(n, dim, K, R, bits, layout, dtype, std_scale=1.0, outlier_every=0, pairing=None, with_prepared=True, uses_tables=True):
    """Decode n vectors (pairing: with the rotary embedding) and compare a sample of rows with the oracle."""
    codes, std_bits, cb, pos = make(n, dim, K, R, std_scale, outlier_every, 7 * n + K + 3 * layout + R)
    cfg = rvq.make_config(dim, 32, layout, R, K, bits, DT[dtype], 0)
    b = rvq.alloc_buffers(cfg, n, cb)
    cd, sd = codes_to_device(cfg, codes), torch.from_numpy(std_bits.view(np.int16)).cuda()
    pos_dev, table = torch.from_numpy(pos).cuda(), None
    if pairing is not None:
        table = torch.empty(POSITIONS, dim // 2, 2, device="cuda")
        rvq.rvq_rope_table(dim, BASE, POSITIONS, table)

    def call(first, count):
        out = torch.full((count, dim + 8), 7.0, dtype=rvq.TORCH_DTYPE[cfg.x_dtype], device="cuda")
        args = (cfg, cd[first * rvq.rvq_code_bytes(cfg):], sd[first:], count, b.codebooks)
        if pairing is None:
            rvq.rvq_decode(*args, b.prepared, out, dim + 8, b.status)
        else:
            rvq.rvq_decode_rope(*args, b.prepared if with_prepared else None, pos_dev[first // HEADS:], HEADS, table, POSITIONS,
                                pairing, out, dim + 8, b.status)
        torch.cuda.synchronize()
        assert torch.all(out[:, dim:] == 7.0)               # row padding untouched
        return out[:, :dim]

    got = call(0, n)
    assert rvq.read_status(b.status)["bad_codes"] == 0
    rows = np.unique(np.concatenate([np.arange(0, n, max(1, n // 9000)), np.arange(max(0, n - 300), n)]))
    values = got[torch.from_numpy(rows).cuda()].float().cpu().numpy().astype(np.float64)
    if pairing is None:
        assert_recon_match(values, codes[rows], std_bits[rows], cb, dim, layout, cfg.x_dtype)
    else:
        ref = oracle.decode_rope(codes[rows], std_bits[rows], cb, pos[rows // HEADS], BASE, pairing, dim, layout)
        # (float32 outputs are float32 sums: at deviations of 40 their ulps come to a few 1e-5, inside the 1e-3)
        assert np.all(np.abs(values - ref) <= RECON_TOL + HALF_ULP[cfg.x_dtype] * np.abs(ref) * 1.01)
    if uses_tables:
        # 16 runs of 2048 vectors, each few enough for the way without tables (16-byte aligned starts)
        direct = torch.cat([call(f, 2048) for f in range(0, 16384, 2048)])
        assert not torch.equal(got[:16384], direct)


# deviations of which most rows are in reach of the summed levels, of the per-stage levels, and of neither; and single rows beyond
KINDS = [(1.0, 0), (4.0, 0), (40.0, 0), (1.0, 97)]


@pytest.mark.parametrize("std_scale,outlier_every", KINDS)
@pytest.mark.parametrize("K,bits,layout,dtype", [(1024, 16, C, "f16"), (1024, 10, S, "bf16"), (1536, 11, C, "bf16"), (1000, 16, S, "bf16"),
                                                 (1100, 11, S, "f16"), (600, 10, C, "f16"), (200, 16, S, "f16")])
def test_four_groups(K, bits, layout, dtype, std_scale, outlier_every):
    run(28677, 128, K, 8, bits, layout, dtype, std_scale, outlier_every)


@pytest.mark.parametrize("std_scale,outlier_every", [(0.3, 0), (2.0, 0), (40.0, 0), (0.3, 97)])
@pytest.mark.parametrize("K,bits,layout,dtype,pairing", [(1024, 16, S, "bf16", rvq.ROPE_HALVES), (1024, 10, C, "f16", rvq.ROPE_HALVES),
                                                         (1536, 11, S, "bf16", rvq.ROPE_ADJACENT), (1000, 16, C, "bf16", rvq.ROPE_ADJACENT),
                                                         (1025, 11, S, "f16", rvq.ROPE_HALVES)])
def test_four_groups_rotated(K, bits, layout, dtype, pairing, std_scale, outlier_every):
    run(131077, 128, K, 8, bits, layout, dtype, std_scale, outlier_every, pairing=pairing)


@pytest.mark.parametrize("n,dim,K,bits,layout,dtype,std_scale,outlier_every", [
    (32771, 256, 1024, 10, C, "bf16", 1.0, 0), (32771, 256, 1024, 16, S, "f16", 1.0, 97), (32771, 256, 1536, 11, S, "bf16", 40.0, 0),
    (32771, 256, 1000, 16, C, "f16", 40.0, 0), (16389, 512, 700, 10, S, "bf16", 1.0, 0),
])
def test_more_groups(n, dim, K, bits, layout, dtype, std_scale, outlier_every):
    run(n, dim, K, 8, bits, layout, dtype, std_scale, outlier_every)


@pytest.mark.parametrize("dim,K,R,bits,layout,dtype,std_scale,outlier_every", [
    (64, 1024, 8, 16, S, "bf16", 1.0, 97), (64, 1536, 8, 11, C, "f16", 40.0, 0), (64, 2048, 8, 11, S, "bf16", 1.0, 97), (64, 3072, 8, 12, C, "f16", 1.0, 0),
    (64, 2048, 6, 16, C, "bf16", 40.0, 0), (64, 1792, 8, 16, C, "f32", 1.0, 0), (64, 3584, 8, 12, S, "f32", 1.0, 0), (64, 3584, 5, 12, C, "bf16", 1.0, 0),
    (64, 1024, 3, 10, S, "f32", 1.0, 0), (32, 1024, 8, 10, C, "bf16", 1.0, 97), (32, 3000, 8, 12, S, "f16", 1.0, 0), (32, 2000, 8, 16, C, "f32", 1.0, 0),
])
def test_one_or_two_groups(dim, K, R, bits, layout, dtype, std_scale, outlier_every):
    run(1531, dim, K, R, bits, layout, dtype, std_scale, outlier_every, uses_tables=False)


@pytest.mark.parametrize("pairing", [rvq.ROPE_HALVES, rvq.ROPE_ADJACENT])
@pytest.mark.parametrize("layout", [C, S])
@pytest.mark.parametrize("K,bits,dtype,std_scale,with_prepared", [(1024, 10, "bf16", 1.0, True), (2048, 11, "bf16", 0.3, True), (3072, 12, "f16", 40.0, True),
                                                                  (3584, 12, "bf16", 1.0, False), (1792, 16, "f32", 1.0, True), (2048, 11, "f32", 1.0, True)])
def test_two_groups_rotated(K, bits, dtype, std_scale, with_prepared, layout, pairing):
    run(1531, 64, K, 8, bits, layout, dtype, std_scale, pairing=pairing, with_prepared=with_prepared, uses_tables=False)
