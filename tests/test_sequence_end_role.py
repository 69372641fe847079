"""The warp of the SM-wide attention kernel that zeroes V's rows past a sequence's end (wpp_attention.cu): how long it stays when a
CTA has no end of a sequence to work on, as a model on the CPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35263_b200", "csrc")


def _role():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "wpp_attention.cu")).read())
    return src[src.index("if (warp == 15)"):src.index("} else if (warp == 13)")]


def _stays(tiles, handed_on, limit, anew):
    """Whether the role is there when the last of `tiles` tiles asks for it, handed on every `handed_on` seconds."""
    now = since = 0.0
    seen = -1
    while now < tiles * handed_on:
        now += limit / 16
        if now - since > limit:
            tile = int(now / handed_on) // 2 * 2               # (of the queue's first place: every second one)
            if not anew or tile == seen:
                return False
            seen, since = tile, now
    return True


def test_the_role_stays_as_long_as_tiles_are_handed_on():
    """A wave on one CTA (max_ctas = 1) may go on for minutes without an end of a sequence."""
    body = _role()
    limit = 64 * 2.0 ** 30 / 1.9e9                             # s
    anew = re.search(r"if \(tile_ids\[0\] == tile\) \{ \*abort_flag = 1u; break; \}\s*tile = tile_ids\[0\];\s*t0 = clock64\(\);", body) is not None
    assert not _stays(4000, 0.02, limit, False)
    assert _stays(4000, 0.02, limit, anew)


def test_every_wait_of_the_role_has_a_limit():
    body = _role()
    assert "64 * WPP_WAIT_LIMIT" in body and "*abort_flag" in body
    assert not _stays(1, 1e9, 36.0, True)                      # no tile is handed on: the limit holds
