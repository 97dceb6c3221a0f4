"""Properties of the kernels' sources that no run can show: a hand-over without its
release half gives the right result on almost every run."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_08684_gb300", "csrc")


def _code(name):
    """The source without its // comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_decode_hands_on_the_zeroed_counters_by_release_and_acquire():
    # The producer acquires the init flag (CTA 0's zeroing of the counters); the
    # consumers count on those counters once they read init_seen, so the word
    # between them is stored with release and read with acquire.
    code = _code("decode.cu")
    uses = [u.strip() for u in re.findall(r"[^;{}]*\binit_seen\b[^;{}]*", code)
            if re.search(r"s\.init_seen", u)]
    stores = [u for u in uses if re.search(r"init_seen\s*=[^=]|st_\w+\(&s\.init_seen", u)]
    # set to 0 before the block's first barrier, then only by a release store
    assert sorted(re.sub(r"\s+", " ", u) for u in stores) == [
        "s.init_seen = 0", "st_release_cta(&s.init_seen, 1)"]
    wait = re.search(r"bool wait_seen\(.*?\n}\n", code, re.S).group(0)
    assert "ld_acquire_cta(seen)" in wait and "volatile int *)seen" not in wait
    # every other use passes the word to that wait
    assert all("wait_seen(p, &s.init_seen" in u for u in uses if u not in stores), uses
