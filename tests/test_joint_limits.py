"""The limits that the joint recurrence tests: each inside the interval that is left, few of them, and the right answer."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_limits_of_any_costs(tmp_path):
    """Costs from 1 to 2^61 ns, crowded towards either end or not, one cost, guesses and bounds that are right, wrong or no cost at all: a
    search whose steps double has to end, whatever the costs are (a launch that did not would hang)."""
    exe = str(tmp_path / "joint_limits")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-o", exe,
                    os.path.join(ROOT, "tests", "joint_limits.cu")], check=True)
    rows = [line.split() for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) > 300
    for name, most, lost, wrong in rows:
        assert (int(lost), int(wrong)) == (0, 0) and int(most) <= 128, (name, most, lost, wrong)
