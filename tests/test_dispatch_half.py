"""Which calls of the weight-only layer take binary16 operands (host-only): sizes on both sides of each line of the rule."""
import pytest

from paper_2203_15952_b200 import binding as aqt

NONE, SWISH, GLU = aqt.ACT_NONE, aqt.ACT_SWISH, aqt.ACT_GLU


@pytest.mark.parametrize("M,N,K,act,half", [
    (12800, 2048, 512, SWISH, True), (1281, 4096, 256, NONE, True), (30000, 1024, 1024, NONE, True),
    # sizes for which the workspace has no room
    (12800, 1016, 512, NONE, False), (1023, 2048, 1024, NONE, False), (12800, 2048, 248, NONE, False), (12800, 2048, 516, NONE, False),
    (12800, 2048, 1032, NONE, False), (1040, 4096, 304, NONE, False),
    # one round of pairs, and of few tiles
    (1614, 2432, 488, NONE, False), (1614, 2432, 496, NONE, True), (1614, 2432, 496, SWISH, True), (3102, 1216, 504, GLU, False),
    (3102, 1216, 512, GLU, True), (1698, 1096, 896, NONE, False), (1100, 1280, 1024, NONE, True), (1024, 2048, 640, NONE, False),
    # epilogues with an activation
    (18359, 1824, 312, SWISH, False), (18359, 1824, 320, SWISH, True), (18359, 1824, 296, NONE, True), (2629, 2440, 408, GLU, False),
    (2629, 2440, 416, GLU, True), (43495, 1528, 344, GLU, False), (43495, 1528, 352, GLU, True), (7122, 3192, 304, aqt.ACT_GLU_SWISH, True),
    # few columns in full rounds
    (31595, 1096, 648, NONE, False), (31595, 1096, 704, NONE, True), (31595, 1152, 648, NONE, True), (15311, 1064, 256, NONE, True),
    (2600, 1024, 512, NONE, True),
    (31324, 1288, 280, NONE, False), (31324, 1344, 280, NONE, True), (31324, 1280, 280, NONE, True)])
def test_line_of_the_binary16_form(M, N, K, act, half):
    plan = aqt.aqt_plan_qmatmul(M, N, K, 0, 4 | aqt.PLAN_WEIGHT_ONLY, act, float_kind=True, sm_count=148)
    assert (plan == "pair256s4e8f16") == half
    if not half:
        assert plan == aqt.aqt_plan_qmatmul(M, N, K, 0, 4, act, float_kind=True, sm_count=148)
    else:  # such a call finds its room in the workspace asked for
        assert aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, M, N, K, 0, 4) >= 4 * N * K + 2 * N * K + 2 * M * K + 4 * M


def test_flags_of_the_plan_query():
    with pytest.raises(aqt.AqtError):
        aqt.aqt_plan_qmatmul(12800, 2048, 512, 8, 4 | aqt.PLAN_WEIGHT_ONLY, sm_count=148)  # of the float kind alone
    assert aqt.aqt_workspace_bytes(aqt.OP_LINEAR_WEIGHT_ONLY, (1 << 31) - 1, (1 << 31) - 4, 1024, 0, 4) > 1 << 41
