"""GPU parity of the table kernels of rvq_attention_decode (caches of more than 28672 tokens, 12288 with up to four stages) at the code widths,
depths and query-head counts that take their own branch."""
import pytest

import paper_2410_15704_b200 as rvq
import rvq_synth
from test_gpu_attention import run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens, q_heads, depths, bits, K, layouts, pairing", [
    (32769, 32, (8, 8), (16, 16), 1024, (rvq_synth.STRIDED, rvq_synth.CONTIGUOUS), rvq.ROPE_HALVES),
    (28672, 32, (8, 8), (16, 16), 256, (rvq_synth.STRIDED, rvq_synth.CONTIGUOUS), rvq.ROPE_HALVES),
    (28673, 8, (8, 4), (16, 16), 256, (rvq_synth.STRIDED, rvq_synth.CONTIGUOUS), rvq.ROPE_HALVES),
    (12288, 16, (4, 4), (8, 8), 256, (rvq_synth.STRIDED, rvq_synth.CONTIGUOUS), rvq.ROPE_HALVES),
    (12289, 16, (4, 3), (9, 16), 300, (rvq_synth.CONTIGUOUS, rvq_synth.STRIDED), rvq.ROPE_HALVES),
    (33001, 8, (6, 8), (10, 16), 1000, (rvq_synth.STRIDED, rvq_synth.CONTIGUOUS), rvq.ROPE_ADJACENT),
    (32769, 32, (5, 4), (16, 8), 256, (rvq_synth.STRIDED, rvq_synth.STRIDED), rvq.ROPE_HALVES),
    (32769, 32, (1, 2), (1, 1), 2, (rvq_synth.STRIDED, rvq_synth.CONTIGUOUS), rvq.ROPE_HALVES),
    (32769, 16, (8, 7), (11, 11), 1752, (rvq_synth.CONTIGUOUS, rvq_synth.CONTIGUOUS), rvq.ROPE_ADJACENT),
])
def test_attention_of_long_caches(tokens, q_heads, depths, bits, K, layouts, pairing):
    run_case(tokens, q_heads, Kk=K, Kv=K, Rk=depths[0], Rv=depths[1], bits_k=bits[0], bits_v=bits[1],
             layout_k=layouts[0], layout_v=layouts[1], pairing=pairing)
