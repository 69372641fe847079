"""The warp of the SM-wide attention kernel that zeroes V's rows past a sequence's end (wpp_attention.cu): what its source has to keep
so that it is there for as long as a CTA may work without such an end."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35263_b200", "csrc")


def _source():
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "wpp_attention.cu")).read())


def _role():
    src = _source()
    return src[src.index("if (warp == 15)"):src.index("} else if (warp == 13)")]


def test_the_role_outlasts_any_launch():
    """A wave of 128 requests takes 148 SMs 0.125 s and one CTA (max_ctas = 1) 18 s: its limit is not to be within a hundred of
    them, for once it has left, the next end of a sequence in that CTA runs out of its wait."""
    limit = int(re.search(r"clock64\(\) - t0 < (\d+) \* WPP_WAIT_LIMIT", _role()).group(1)) * 2.0 ** 30 / 1.965e9
    assert limit > 100 * 148 * 0.125


def test_the_role_is_told_when_there_is_no_more_and_when_a_wait_was_given_up():
    assert "!*abort_flag" in _role()
    src = _source()
    issuer = src[src.index("dead = false", src.index("idesc_pv")):]
    body, bye = issuer[:issuer.index("v_rows[0] = -1;")], issuer[issuer.index("v_rows[0] = -1;"):]
    assert "return" not in body                                # every way out of the issuing thread's loop comes here
    assert re.match(r"v_rows\[0\] = -1;\s*mbar_arrive\(bVAsk\);", bye)
