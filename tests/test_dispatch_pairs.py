"""Where 8-bit matmuls change to pairs of CTAs, and between the pair configurations."""
import pytest

from paper_2203_15952_b200 import binding as aqt
from paper_2203_15952_b200 import inputs as gen


@pytest.mark.parametrize("M,N,K,act,plan", [
    (23 * 256, 512, 2048, gen.ACT_NONE, "stream64s5e8"), (23 * 256 + 1, 512, 2048, gen.ACT_NONE, "pair256s4e8"),  # 46 and 48 pair tiles
    (9472, 512, 2048, gen.ACT_NONE, "pair256s4e8"), (9473, 512, 2048, gen.ACT_NONE, "pair512s3e16"),   # one round of pairs, and more
    (14080, 512, 2048, gen.ACT_NONE, "pair512s3e16"), (14081, 512, 2048, gen.ACT_NONE, "pair256s4e8"),  # a second round half full
    (12800, 2048, 1024, gen.ACT_NONE, "pair256s4e8"), (12800, 2064, 1024, gen.ACT_NONE, "stream128s4e16"),
    (12544, 2064, 2048, gen.ACT_NONE, "pair256s4e8"),                                                  # any width from K = 2048
    (12800, 1024, 512, gen.ACT_NONE, "ws128e16"), (12800, 1024, 528, gen.ACT_NONE, "pair256s4e8"),
    (74 * 256, 256, 1024, gen.ACT_NONE, "pair256s4e8"), (81 * 256, 256, 1024, gen.ACT_NONE, "pair128s6e8"),  # a last round of 7 of 74
    (82 * 256, 256, 1024, gen.ACT_NONE, "pair256s4e8"),
    (18944, 2048, 2048, gen.ACT_SWISH, "pair256s4e8"), (4000, 2048, 2048, gen.ACT_SWISH, "stream256s3e16"),
])
def test_cta_pairs_start_and_end_where_the_rules_say(M, N, K, act, plan):
    """Both sides of each line in the choice of CTA pairs for 8-bit matmuls (sizes that other tests run by plan name)."""
    assert aqt.aqt_plan_qmatmul(M, N, K, 8, aqt.BITS_4_UNPACKED, act, sm_count=148) == plan


@pytest.mark.parametrize("M,N,K,act,plan", [
    # one tile column of 128: single CTAs in the first round of pairs, else pairs of 128 columns
    (74 * 256, 128, 4096, gen.ACT_NONE, "stream128s4e16"), (74 * 256 + 1, 128, 1024, gen.ACT_NONE, "pair128s6e8"),
    (30000, 128, 528, gen.ACT_NONE, "pair128s6e8"), (30000, 144, 1008, gen.ACT_NONE, "pair256s4e8"),
    # from K = 4096 pairs as soon as 128-column tiles of single CTAs take a second round, with Swish as soon as pairs do
    (37 * 128 + 1, 512, 4096, gen.ACT_NONE, "pair256s4e8"), (37 * 128, 512, 4096, gen.ACT_NONE, "stream128s4e16"),
    (37 * 128 + 1, 512, 4080, gen.ACT_NONE, "stream64s5e8"),
    (4000, 1536, 4096, gen.ACT_SWISH, "pair256s4e8"), (4000, 1536, 4080, gen.ACT_SWISH, "stream128s4e16"),
    (37 * 256, 512, 4096, gen.ACT_SWISH, "stream256s3e16"),
    # a last round of 6 of 74: 256 columns where the tiles are deep and full
    (5000, 1024, 4096, gen.ACT_NONE, "pair256s4e8"), (5000, 1024, 4080, gen.ACT_NONE, "pair128s6e8"), (20 * 256, 1000, 4096, gen.ACT_NONE, "pair128s6e8"),
    (20000, 256, 4096, gen.ACT_NONE, "pair128s6e8"),
])
def test_cta_pairs_of_deep_and_of_narrow_matmuls(M, N, K, act, plan):
    """Both sides of the lines for one column of 128-wide tiles and for K from 4096."""
    assert aqt.aqt_plan_qmatmul(M, N, K, 8, aqt.BITS_4_UNPACKED, act, sm_count=148) == plan


@pytest.mark.parametrize("M,N,K,act,plan", [
    # from 32 pair tiles, below K = 1024 from the 38th on (K in elements)
    (4096, 512, 1024, gen.ACT_NONE, "pair128s6e8"), (31 * 256, 256, 1024, gen.ACT_NONE, "stream128s4e16"),
    (4096, 512, 1020, gen.ACT_NONE, "stream128s4e16"), (38 * 256, 256, 1020, gen.ACT_NONE, "pair256s4e8"),
    # a last round of pairs that is nearly empty counts beyond K = 512
    (7000, 2048, 512, gen.ACT_NONE, "pair256s4e8"), (7000, 2048, 516, gen.ACT_NONE, "stream256s4e8"), (7000, 2048, 2048, gen.ACT_NONE, "stream256s4e8"),
    # below K = 512: one column of 128 from the second round on, with an activation from the third; Swish with padding from the second
    (74 * 256, 128, 508, gen.ACT_NONE, "stream128s4e16"), (75 * 256, 128, 508, gen.ACT_NONE, "pair128s6e8"), (38 * 256, 128, 512, gen.ACT_NONE, "pair128s6e8"),
    (148 * 256, 128, 508, gen.ACT_SWISH, "stream128s4e16"), (149 * 256, 128, 508, gen.ACT_SWISH, "pair128s6e8"), (7000, 384, 160, gen.ACT_SWISH, "pair256s4e8"),
    (7000, 320, 160, gen.ACT_SWISH, "stream64s5e8"), (7000, 320, 160, gen.ACT_NONE, "pair256s4e8"), (9473, 320, 160, gen.ACT_SWISH, "pair128s6e8"),
    (7000, 320, 512, gen.ACT_SWISH, "pair256s4e8"),
    # width: 0.7 of a round of 256 columns, 0.6 below K = 512 without a gate
    (20000, 320, 1024, gen.ACT_NONE, "pair128s6e8"), (20000, 320, 2048, gen.ACT_SWISH, "pair128s6e8"), (25600, 1024, 1024, gen.ACT_NONE, "pair256s4e8"),
    (32768, 320, 160, gen.ACT_NONE, "pair128s6e8"), (32768, 320, 160, gen.ACT_GLU, "pair256s4e8"), (32768, 320, 512, gen.ACT_NONE, "pair256s4e8"),
    (65536, 640, 256, gen.ACT_GLU, "pair256s4e8"), (9500, 384, 4096, gen.ACT_NONE, "pair128s6e8"), (65536, 1152, 4096, gen.ACT_NONE, "pair256s6e4"),
])
def test_cta_pairs_of_the_float_kind(M, N, K, act, plan):
    """Both sides of each line in the choice for float activations; beyond K = 128 elements, where the weights do not stay."""
    assert aqt.aqt_plan_qmatmul(M, N, K, 0, 4, act, float_kind=True, sm_count=148) == plan
