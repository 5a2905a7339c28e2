"""The bench line's flop count against the committed ncu capture of the x pass (CPU): a launch
cannot do more arithmetic than its FMA pipe was active for."""
import re
import sys
from pathlib import Path

ROOT = Path(__file__).resolve().parents[1]
sys.path.insert(0, str(ROOT))


def test_counted_flops_fit_the_fma_pipe():
    import bench

    text = (ROOT / "profiles" / "k_xpass_full_twinned128_fp32.md").read_text()
    ms = float(re.search(r"duration \(ms[^|]*\| ([\d.]+)", text).group(1))
    active = float(re.search(r"FMA pipe cycles active \(%\) \| ([\d.]+)", text).group(1)) / 100
    peak = 152 * 128 * 2 * 2070.0e6  # flop/s of the FMA pipe
    rate = bench.flops_per_voxit(bench.N_SUB) * 128**3 / (ms * 1e-3)
    assert rate <= active * peak, (rate / peak, active)
