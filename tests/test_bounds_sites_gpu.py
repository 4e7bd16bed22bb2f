"""The bounds-checked build: the guard of every array of the paired lines' path
stands where the array is accessed.  A test hook makes the guard at one site
report every access and skip it; the call must then return SGM_EDEVICE and name
the site.  Nothing is read or written out of range.  The checked library runs in
a child process (SGM_BOUNDS_CHECK=1 selects it in the binding).
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# site -> the call that passes it
SITES = {301: "plain", 302: "plain", 306: "plain", 308: "plain", 309: "per_line", 310: "plain", 311: "post", 312: "post",
         313: "plain", 314: "mirror", 315: "post", 316: "post", 317: "post", 101: "plain", 102: "plain", 103: "plain",
         104: "post", 105: "plain", 106: "plain", 111: "plain", 112: "plain", 113: "plain", 114: "plain", 115: "plain",
         116: "plain", 117: "post", 118: "plain4", 119: "post", 120: "debug"}

SCRIPT = """
import sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_1610_04121_gb300 import sgm
assert sgm.sgm_bounds_checked()
rng = np.random.default_rng(1)
left, right = (rng.integers(0, 256, (41, 77), dtype=np.uint8) for _ in range(2))
calls = dict(plain=lambda c: c.compute(left, right, 64, 7, 84, 8), plain4=lambda c: c.compute(left, right, 64, 7, 84, 4),
             per_line=lambda c: c.compute(left, right, 64, 7, 84, 4), post=lambda c: c.compute_ex(left, right, 64, 7, 84, 8, 7),
             mirror=lambda c: c.compute_ex(left, right, 64, 7, 84, 8, 2), debug=lambda c: c.debug(left, right, 64, 7, 84, 8))
# a cap that holds the per-line sweeps' arena and not two passes' cubes
cap = 41 * 77 * (7 * 64 + 20) + 3 * 77 * 64 * 4 * 4 + 4096 if {call!r} == "mirror" else 0
with sgm.Context(0, mem_cap_bytes=cap) as c:
    sgm.sgm_set_schedule(c.handle, sgm.SGM_SCHED_V_THEN_H if {call!r} == "per_line" else sgm.SGM_SCHED_PAIRS)
    try:
        calls[{call!r}](c)
        raise SystemExit("no guard fired")
    except sgm.SgmError as e:
        assert e.code == sgm.SGM_EDEVICE and "site {site}" in str(e), e
print("ok")
"""


@pytest.fixture(scope="module")
def checked_lib():
    from paper_1610_04121_gb300 import build

    return build.build(bounds_check=True)


@pytest.mark.parametrize("call", sorted(set(SITES.values())))
def test_the_guard_of_every_site_is_on_its_path(checked_lib, call):
    missing = []
    for site in sorted(s for s, v in SITES.items() if v == call):
        r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT, call=call, site=site)], cwd=ROOT,
                           env=dict(os.environ, SGM_BOUNDS_CHECK="1", SGM_TEST_BOUNDS_SITE=str(site)),
                           capture_output=True, text=True, timeout=300)
        if r.returncode != 0 or not r.stdout.strip().endswith("ok"):
            missing.append((site, (r.stdout + r.stderr)[-300:]))
    assert not missing, missing
