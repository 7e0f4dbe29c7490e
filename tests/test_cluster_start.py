"""Distributed shared memory is only touched while every CTA of the cluster runs.

A CTA may access another one's shared memory only between a cluster barrier that
shows the other has started and one that holds the other's exit back.  A race on
this cannot be provoked reliably, so the kernels' sources are read: with the calls
of device functions expanded in place, every kernel that uses
``map_shared_rank`` has to pass a cluster barrier before its first access and
another one after its last.
"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1208_4093_gb300", "csrc")
BARRIER = r"\b\w+\.sync\(\)|\bcluster_wait\(\)"
MAPPED = r"[*&]?\s*\b\w+\.map_shared_rank\("


def strip_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def closing(text, at, pair):
    depth = 0
    for k in range(at, len(text)):
        depth += (text[k] == pair[0]) - (text[k] == pair[1])
        if depth == 0:
            return k
    raise ValueError("unbalanced")


def functions(text):
    """name -> (is a kernel, body) of the device functions and kernels."""
    out = {}
    for m in re.finditer(r"__(global|device)__\b", text):
        if re.match(r"\s*const\s+\w+(<[^<>]*>)?\s+\w+\s*=", text[m.end():]):
            continue  # a constant table
        head = re.compile(r"([A-Za-z_]\w*)\s*\(").finditer(text, m.end())
        name = next(h for h in head if not h.group(1).startswith("__"))
        args = closing(text, name.end() - 1, "()")
        brace = re.compile(r"\s*([{;])").match(text, args + 1)
        if brace and brace.group(1) == "{":
            end = closing(text, brace.start(1), "{}")
            kernel, body = out.get(name.group(1), (False, ""))  # specialisations of one name together
            out[name.group(1)] = (kernel or m.group(1) == "global", body + text[brace.start(1):end])
    return out


def events(name, funcs, seen=()):
    """Barriers and remote accesses of a function in the order of its text."""
    body = funcs[name][1]
    at = [(m.start(), ["barrier"]) for m in re.finditer(BARRIER, body)]
    for m in re.finditer(MAPPED, body):
        # a pointer that is only kept is an access where it is used next
        keep = None if m.group(0)[0] in "*&" else re.search(r"(\w+)(?:\[\w+\])?\s*=\s*$", body[:m.start()])
        end = body.find(";", m.end())
        if keep is None:
            at.append((m.start(), ["remote"]))
        else:
            at += [(end + u.start(), ["remote"]) for u in re.finditer(r"\b%s\b" % keep.group(1), body[end:])]
    for f in funcs:
        if f not in seen and f != name:
            at += [(m.start(), events(f, funcs, seen + (name,)))
                   for m in re.finditer(r"\b%s\s*(?:<[^;(){}]*>)?\s*\(" % f, body)]
    return [e for _, es in sorted(at, key=lambda t: t[0]) for e in es]


def wrong(text):
    funcs = functions(strip_comments(text))
    bad = []
    for name, (kernel, _) in funcs.items():
        ev = events(name, funcs) if kernel else []
        if "remote" in ev and (ev[0] != "barrier" or ev[-1] != "barrier"):
            bad.append(name)
    return bad


def test_the_reader_sees_a_missing_barrier():
    body = "__device__ void put(int* p) { *cluster.map_shared_rank(p, 1) = 3; }\n"
    kernel = "__global__ void __launch_bounds__(32) k(int* p) { %s put(p); %s }"
    start, end = "cluster_wait();", "cluster.sync();"
    assert wrong(body + kernel % (start, end)) == []
    assert wrong(body + kernel % ("", end)) == ["k"]
    assert wrong(body + kernel % (start, "")) == ["k"]
    kept = "__global__ void k(int* p) { int* q = cluster.map_shared_rank(p, 1); %s q[0] = 1; cluster.sync(); }"
    assert wrong(kept % "cluster.sync();") == [] and wrong(kept % "") == ["k"]


def test_remote_accesses_lie_between_cluster_barriers():
    users = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        users += "map_shared_rank" in strip_comments(text)
        assert wrong(text) == [], os.path.basename(path)
    assert users >= 4  # slots, tree of fronts, band factors: the files were read
