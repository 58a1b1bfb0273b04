"""The small-batch blind rotation when words do not arrive: each CTA's wait ends at
its limit, the kernel ends, TIMEOUT is reported once, and the context goes on."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _libs():
    from paper_2609_16915_gb300 import build
    build.build()
    build.build(debug=True)


def test_lost_words_end_in_a_timeout_and_the_context_stays_usable():
    r = subprocess.run([sys.executable, "-m", "tests.lost_words_client"], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(res) == 40
    assert all(v == [-6, 0, True] for v in res.values()), res


def test_regular_build_has_no_such_switch():
    import paper_2609_16915_gb300 as R
    import workload as W
    ctx = R.Context(W.CONFIGS["tiny"])
    with pytest.raises(R.RosettaError) as e:
        ctx.selftest_lost_words()
    assert e.value.status == -2
    ctx.close()
