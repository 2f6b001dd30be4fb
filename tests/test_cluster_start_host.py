"""Clusters: no block's shared memory is accessed before that block is known to run.

Read from the sources, since a run cannot show a missing wait: the blocks of a
cluster are launched together and an access microseconds later finds them
running, but only a cluster barrier says so. Rules (launch.cuh): a kernel that
uses cluster_at, itself or in a function it calls, first calls cluster_arrive and
then, before the first use, cluster_running; nothing else maps another block's
shared memory.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2306_07603_gb300", "csrc")


def _functions(text):
    """(name, body) of every function definition of a source (braces matched, comments gone)."""
    text = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))
    for m in re.finditer(r"(\w+)\s*\(([^;{}()]*)\)\s*\{", text):
        if m.group(1) in ("if", "for", "while", "switch"):
            continue
        depth, k = 1, m.end()
        while depth and k < len(text):
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), text[m.end():k]


def test_cluster_memory_is_accessed_only_after_the_start_barrier():
    users = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        if os.path.basename(path) == "launch.cuh":
            continue
        assert "map_shared_rank" not in text and "mapa" not in text, path
        funcs = dict(_functions(text))
        inner = {n for n, b in funcs.items() if "cluster_at<" in b and "cluster_arrive<" not in b}
        for name, body in funcs.items():
            called = [n for n in inner if n != name and re.search(r"\b%s\s*<" % n, body)]
            # a helper that uses cluster_at is judged within the kernel that calls it
            for n in called:
                if "cluster_arrive<" not in body:
                    # the single-block form: cluster_at is the block's own memory
                    assert re.findall(r"\b%s\s*<\s*(\w+)" % n, body) == ["1"], (path, name)
                    continue
                body = re.sub(r"\b%s\s*<.*" % n, lambda _: funcs[n], body, flags=re.S)
            if name in inner or "cluster_at<" not in body:
                continue
            users += 1
            a, w, u = (body.find(t) for t in ("cluster_arrive<", "cluster_running<", "cluster_at<"))
            assert 0 <= a < w < u, (path, name)
            assert body.find("cluster_done<") > u, (path, name)
        for n in inner:
            assert 0 <= funcs[n].find("cluster_running<") < funcs[n].find("cluster_at<"), (path, n)
    assert users == 3      # the residual, the fields and the adjoint's parameters
