"""Every kernel that selects, at sizes that the dispatch gives it (the test looks at what was launched): the orders of the
lists, crowded bins, ties, infinities.  Scores are exact, the lists are the oracle's."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_parity import H  # noqa: E402,F401
from test_gpu_select_stream import check_lists  # noqa: E402


# Crowded bins, thresholds above and below the sampled bracket, lists too short for a sample, ties, infinities.
HARD = ["int", "ties", "outliers", "below", "binades", "infs"]


def hard(heads, g, lens, dp, dtype, reduce, budget, sinks=0, recent=0, radius=0, mode=0):
    budgets = {"outliers": 40, "below": 9 * max(lens) // 20}
    return [(heads, g, lens, dp, dtype, reduce, budgets.get(data, budget), sinks, recent, radius, mode, data) for data in HARD]


# heads, group, lengths, d', dtype, reduce, budget, sinks, recent, radius, mode, data
@pytest.mark.parametrize("kernel,dev,case", [(kernel, dev, case) for kernel, dev, cases in [
    # more lists than two per SM, between what fits on chip and what is worth two waves of streaming blocks
    ("select_wave", False, hard(8, 1, [5050] + [5040, 2100] * 18 + [700], 32, "bf16", "sum", 400, 2, 31)),
    ("select_wave", False, hard(8, 4, [9999] + [1501, 2048] * 18 + [64], 16, "fp32", "max", 300, 0, 0, 1)),
    # lists that share a key stream, many and long, or under device lengths
    ("select_shared", False, hard(4, 4, [15003] + [14001] * 8 + [700], 32, "bf16", "per head", 600, 3, 5)),
    ("select_shared", False, hard(4, 7, [14100] * 6, 16, "bf16", "per head", 600, 0, 0, 1, 1)),
    ("select_shared", True, hard(2, 4, [12345, 8300], 32, "bf16", "per head", 1000, 0, 0)),
    # a cluster per list on TMA rings: a little more lists than SMs, beyond what one block keeps on chip
    ("select_kernel", True, hard(8, 1, [20603] + [20500, 21000] * 8 + [700, 2100], 32, "bf16", "sum", 777, 5, 9)),
    ("select_kernel", False, hard(8, 1, [31007] + [30000] * 18, 16, "fp32", "sum", 1500)),
    # ... with the keys in the workspace: digits on chip, and beyond
    ("select_cw", False, hard(1, 2, [430001, 400000], 32, "bf16", "sum", 2500, 3, 40, 1)),
    ("select_cw", False, hard(1, 1, [1100001], 16, "bf16", "max", 9000)),
    ("select_cw", False, hard(1, 1, [1060003], 32, "fp32", "sum", 9000)),
] for case in cases])
def test_unusual_distributions(H, kernel, dev, case):
    check_lists(H, case, 3, kernel=kernel, dev_lengths=dev)


# heads, group, lengths, d', dtype, reduce, budget, sinks, recent, radius, mode, data
@pytest.mark.parametrize("kernel,case", [
    # neighbours: one block per list up to 16384 candidates, also of lists that share a key stream, unless these are many
    ("select_small", (8, 4, [16384] + [9001] * 19, 32, "bf16", "sum", 900, 0, 0, 1, 0, "int")),
    ("select_small", (8, 1, [16384, 8300] * 18, 16, "bf16", "max", 500, 0, 0, 2, 1, "int")),
    ("select_small", (8, 4, [16384], 32, "bf16", "per head", 900, 0, 0, 1, 1, "int")),
    ("select_small", (8, 4, [12288] + [9999] * 4, 32, "bf16", "per head", 900, 0, 0, 1, 0, "ties")),
    ("select_shared", (8, 4, [12289] + [9999] * 4, 32, "bf16", "per head", 900, 0, 0, 1, 0, "ties")),
    ("select_wave", (8, 1, [16385, 8300] * 10, 32, "bf16", "sum", 900, 0, 0, 1, 0, "int")),
    ("select_wave", (8, 1, [2050] * 20, 32, "fp32", "sum", 200, 0, 0, 1, 0, "int")),
    ("select_wave", (8, 1, [1000, 300] * 19, 16, "fp32", "sum", 100, 0, 0, 1, 0, "int")),
    ("select_stream", (8, 1, [10300], 32, "bf16", "sum", 900, 0, 0, 1, 0, "int")),
])
def test_lists_under_device_lengths(H, kernel, case):
    check_lists(H, case, 11, kernel=kernel, dev_lengths=True)
