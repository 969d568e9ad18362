"""Hand-overs between the two CTAs of a pair, as the source states them: what one CTA has read or written before it arrives on a barrier
of the other one is ordered by a scope that holds both of them, or by a fence that does."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _code(name):
    text = open(os.path.join(ROOT, "paper_2607_18002_b200", "csrc", name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _uses(name, word):
    """Names of the functions that are given the barriers `word`."""
    return set(re.findall(r"(\w+)\((?:c, )?(?:map_to_cta\()?(?:leader \? )?&sc->" + word + r"\[", _code(name)))


def test_a_ring_slot_is_given_back_by_a_release_to_the_cluster():
    assert _uses("moe_run_pair.cu", "iempty") == {"mbar_init", "mbar_arrive", "mbar_arrive_cluster", "wwait_cluster"}
    # the roles of the second CTA meet on a barrier of their own
    assert _uses("moe_run_pair.cu", "iread") == {"mbar_init", "wait_info"}
    assert "mbar_arrive(leader ? &sc->iempty[islot] : &sc->iread[islot]);" in _code("moe_run_pair.cu")
