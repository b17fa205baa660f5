"""Every polling loop of the kernels is bounded and reports: where it gives up it records ESC_DEV_TIMEOUT, so that
esc_convattn_device_status() cannot return 0 for a launch that carried on without what it waited for."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parents[1] / "paper_2503_06671_b200" / "csrc"
AFTER = 6            # lines between the pause of a loop and the end of what follows where it gives up


def polling_loops():
    for path in sorted(CSRC.glob("*.cu*")):
        lines = path.read_text().splitlines()
        for n, line in enumerate(lines):
            if "__nanosleep(" in line:
                yield path.name, n + 1, "\n".join(lines[max(0, n - 3):n + 1 + AFTER])


def test_polling_loops_are_bounded_and_report():
    loops = list(polling_loops())
    assert len(loops) >= 4
    for name, line, text in loops:
        assert re.search(r"k(Poll|Spin)Limit|kFlagPolls", text), f"{name}:{line}: no bound"
        assert "kDevTimeout" in text, f"{name}:{line}: gives up without a record"
