"""Rules of the CUDA sources whose violation is a race, which no run shows reliably: read from the
text of the kernels, on the CPU."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1501_04552_gb300", "csrc")


def source(name):
    """a source file without its comments"""
    text = open(os.path.join(CSRC, name), encoding="utf-8").read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)


def body(text, head):
    """the braces after the first match of `head`"""
    at = text.index("{", re.search(head, text).end() - 1)
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
    raise AssertionError("unbalanced braces after %s" % head)


def test_finaliser_reads_the_run_state_before_it_advances():
    """finalise(): thread 0 advances the level after the update, and whether a level records decides
    which threads reach the barriers of the reductions.  So every thread reads that decision once,
    ahead of the branches, and a barrier that all threads reach stands before the advance.  The other
    branches leave alone what the decision is made of."""
    text = source("kg_kernels.cuh")
    fin = body(text, r"void finalise\(")
    assert fin.count("kg_recording(dev)") == 1
    assert not re.search(r"\bif\b|fin_reduce|state_after", fin[:fin.index("kg_recording(dev)")])
    last = fin[fin.rindex("else {"):]
    assert "state_after_z" in last and fin.count("state_after_z") == 1
    statements = [" ".join(x.split()) for x in last.strip("else {}\n ").split(";") if x.strip()]
    assert statements[-2] == "__syncthreads()" and statements[-1].startswith("if (threadIdx.x == 0) state_after_z(")
    writes = set(re.findall(r"dev->(\w+)\s*(?:=|\+=|\^=)[^=]", body(text, r"void state_after_x\(") + fin))
    assert not writes & {"level", "energy_every", "complex_field"}, writes


def test_ensemble_bodies_claim_nothing_read_only():
    """The bodies of the ensemble's passes run many times in one launch on arrays that earlier
    passes of it, on other SMs, have written.  Only the tables are read-only there: no other
    pointer may be const __restrict__, which lets loads go past the coherent path."""
    text = source("kg_kernels.cuh") + source("kg_ensemble.cuh")
    called = body(source("kg_ensemble.cuh"), r"void ens_x\(") + body(source("kg_ensemble.cuh"), r"void ens_y\(") + \
        body(source("kg_ensemble.cuh"), r"void ens_z\(")
    bodies = {n for n in re.findall(r"\b(\w+_body)<", called)} | {"x_pair_load", "x_pair_unpack", "ens_x", "ens_y", "ens_z"}
    assert {"x_pair_body", "x_line_body", "col_body", "z_body"} <= bodies
    for name in sorted(bodies):
        args = re.search(r"void %s\((.*?)\)\s*\{" % name, text, re.S).group(1)
        for a in re.split(r",(?![^<]*>)", " ".join(args.split())):
            if "__restrict__" in a and a.strip().startswith("const "):
                assert re.search(r"\b(tw|coef)$", a), (name, a)
