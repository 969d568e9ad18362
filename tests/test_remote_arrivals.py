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


def test_a_stored_tile_is_handed_over_at_cluster_scope():
    code, ptx = _code("moe_run_pair.cu"), _code("moe_ptx.cuh")
    # behind the fence of the warps that count, a relaxed arrival that the other CTA's wait can meet; behind no fence, a release
    assert _uses("moe_run_pair.cu", "done") == {"mbar_init", "arrive_at_leader", "signal_leader", "wwait_cluster"}
    body = lambda text, name: re.search(name + r"\([^)]*\) \{(.*?)\n\}", text, re.S).group(1)
    assert "mbar_arrive_relaxed(map_to_cta(bar, 0))" in body(code, "void signal_leader")
    assert "mbar_arrive_cluster(map_to_cta(bar, 0))" in body(code, "void arrive_at_leader")
    assert body(_code("moe_sched.cuh"), "void count_stored").strip().startswith("fence_acq_rel_gpu();")
    # every arrival on a barrier of the other CTA says what it orders and for whom; one of them is for this CTA: gathered rows
    assert set(re.findall(r"mbarrier\.arrive(\S*)\.shared::cluster\.b64 _, \[%0\];", ptx)) == {".release.cluster", ".relaxed.cluster", ".release.cta"}
    assert re.findall(r"mbar_arrive_remote\((.*?)\);", code) == ["map_to_cta(&sc->full[stage], 0)"]


def test_a_drained_accumulator_is_handed_back_between_tcgen05_fences():
    code = _code("moe_run_pair.cu")
    assert _uses("moe_run_pair.cu", "tempty") == {"mbar_init", "signal_leader", "wwait_relaxed"}
    assert re.search(r"wwait_relaxed\(c, &sc->tempty.*\n\s*tc_fence_after\(\);", code)
    arrivals = re.findall(r"(.*)\n(.*)\n.*signal_leader\(&sc->tempty", code)
    assert len(arrivals) == 2 and all("tc_fence_before" in a and "__syncwarp" in b for a, b in arrivals)
    assert ".relaxed.cluster" in re.search(r"mbar_try_relaxed.*?mbarrier\.try_wait\.parity(\S*) ", _code("moe_ptx.cuh"), re.S).group(1)
