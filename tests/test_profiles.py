"""The profiles' commands: on the 720M-shaped set (tens of GB on the device,
kernels of milliseconds) only launch durations are collected, which ncu takes
in one pass with nothing saved or restored; every other counter comes from a
small case (the 4-layer set of the same shapes, the 124M-shaped set)."""

import os
import re

PROFILES = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "profiles")
FULL_SIZE = re.compile(r"720m(?!_4layers)", re.IGNORECASE)


def _ncu_commands(text):
    """Every command with ncu in it, continuation lines joined."""
    out, cur = [], ""
    for line in text.splitlines():
        line = line.lstrip("# ").strip()
        cur += " " + line.rstrip("\\&").strip()
        if not line.endswith(("\\", "&&")):
            if "ncu " in cur and "--clock-control" in cur:
                out.append(re.sub(r"(-o|--log-file) \S+|> \S+", "", cur))   # names of outputs
            cur = ""
    return out


def test_no_counters_on_the_full_size_set():
    seen = 0
    for name in sorted(os.listdir(PROFILES)):
        for cmd in _ncu_commands(open(os.path.join(PROFILES, name)).read()):
            seen += 1
            metrics = re.search(r"--metrics (\S+)", cmd)
            options = cmd.split("ncu ", 1)[1].split("python")[0]   # (bench.py has a --set of its own)
            duration_only = (metrics is not None and metrics.group(1) == "gpu__time_duration.sum"
                             and "--set " not in options and "--section" not in options)
            default_set = "bench.py" in cmd and "--set " not in cmd   # the benchmark's default is the 720M set
            assert duration_only or not (FULL_SIZE.search(cmd) or default_set), (name, cmd)
    assert seen >= 4
