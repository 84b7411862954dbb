"""lsms_get_option gives back what lsms_set_option set, so saving an option and restoring it changes nothing:
"streams" is 0 (by the chunk's size, or the environment variable) until it is set."""
import json
import os
import subprocess
import sys

import pytest

from ._util import ROOT, ensure_built

OPTIONS = {"growth_limit": 1e3, "fallback_slots": 8, "ir_max_sweeps": 6, "streams": 0, "residual_tc": 1,
           "solve_cols": 0, "solve_regs": 0, "nvtx": 0, "solve_steps": 0}


@pytest.mark.parametrize("env", [None, "2"])
def test_save_and_restore_is_neutral(env):
    ensure_built()
    code = f"""
import json
from paper_2311_12134_gb300 import autotune as at, binding as B
names = {sorted(OPTIONS)!r}
first = {{k: B.get_option(k) for k in names}}
for k, v in first.items():
    B.set_option(k, v)
at.apply({{k: B.get_option(k) for k in at.DEFAULTS}})
B.set_option("streams", 3)
three = B.get_option("streams")
B.set_option("streams", first["streams"])
print(json.dumps([first, {{k: B.get_option(k) for k in names}}, three]))
"""
    e = dict(os.environ)
    e.pop("LSMS_STREAMS", None)
    if env:
        e["LSMS_STREAMS"] = env
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=e, capture_output=True, text=True, check=True)
    first, last, three = json.loads(r.stdout.splitlines()[-1])
    assert first == last == OPTIONS and three == 3
