"""Waits between the roles of a kernel are bounded: a warp may leave its loop when a wait runs out, so no other warp may wait for it
on a barrier without a limit.  Named barriers (which have none) are for code in which nobody can have left."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_10103_b200", "csrc")

# file: named barriers, and why nobody can be missing there
NAMED = {
    "k_swa_mma.cuh": 1,     # a unit's warps: no role of it has a wait that can run out
    "k_swa_tc5.cuh": 1,     # the second pass: entered by all its threads, after the roles have met and none has given up
}
# barriers of a whole cluster: arrive and wait
CLUSTER = {
    "k_pool_select.cuh": 2,     # every thread of every thread block reaches them: nothing in front of them can run out or leave
}


def sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def test_no_named_barrier_between_roles():
    found = {f: len(re.findall(r"\b(?:bar|barrier)(?:\.cta)?\.(?:sync|arrive|red)", s)) for f, s in sources().items()}
    assert {f: n for f, n in found.items() if n} == NAMED


def test_no_cluster_barrier_behind_a_way_out():
    found = {f: len(re.findall(r"\bbarrier\.cluster\.(?:arrive|wait)", s)) for f, s in sources().items()}
    assert {f: n for f, n in found.items() if n} == CLUSTER
    for f, s in sources().items():
        s = re.sub(r"__forceinline__ void cluster_\w+\(\)", "", s)                   # (the definitions)
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\([^{;]*\{", s, re.S):
            body = s[m.end():s.find("\n}\n", m.end())]
            if "cluster_arrive()" not in body and "cluster_wait()" not in body:
                continue
            assert f in CLUSTER and "mbar_" not in body and "while" not in body, m.group(1)
            last = max(body.rfind("cluster_arrive()"), body.rfind("cluster_wait()"))
            assert "return" not in body[:last], m.group(1)


def test_every_polling_loop_has_a_limit():
    for f, s in sources().items():
        for m in re.finditer(r"while \(!mbar_try_wait[^;{]*", s):
            assert "clock64() - t0 <" in m.group(0), f"{f}: {m.group(0)}"


def test_second_pass_is_behind_every_output_store():
    """A bulk store is complete for the thread that issued it: each warp of the attention kernel that stores output has to wait itself,
    in front of a barrier of the whole thread block, before rows are written a second time by other threads."""
    s = sources()["k_swa_tc5.cuh"]
    end = s[s.index("const int n_redo"):]
    wait, meet, leave = (end.index(x) for x in ("if (warp < C::NSW && lane == 0) bulk_wait_all();", "__syncthreads();", "threadIdx.x >= 256"))
    assert wait < meet < leave < end.index("swa_redo_unit<")
