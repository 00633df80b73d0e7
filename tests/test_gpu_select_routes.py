"""Every kernel that selects, at sizes that the dispatch gives it (the test looks at what was launched): the orders of the
lists, crowded bins, ties, infinities.  Scores are exact, the lists are the oracle's."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_parity import H  # noqa: E402,F401
from test_gpu_select_stream import check_lists  # noqa: E402


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
