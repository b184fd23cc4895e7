"""The batched dataflow passes wait on tags inside the data, so what a tag speaks for has to be one single-copy atomic
element: a (hi, lo) pair is loaded and stored as 64 bits, relaxed at GPU scope, and nothing that a warp of another block
waits on is written by a weak store.  A torn pair needs two SMs and bad luck to show, so the source is what is checked."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_03778_gb300", "csrc",
                   "kern_flowb.cu")


def functions(text, name):
    """(parameters, body) of every definition of a function template"""
    for m in re.finditer(r"\b%s\(([^)]*)\)\s*\{" % name, text):
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        yield m.group(1), text[m.end():at]


def test_pairs_are_single_elements():
    text = open(SRC).read()
    for name, kind in (("ld_row", "ld"), ("put_row", "st")):
        seen = set()
        for params, body in functions(text, name):
            ops = re.findall(r'"((?:ld|st)\.[\w.]+)', body)
            assert len(ops) == 3 and all(o.startswith(f"{kind}.relaxed.gpu.global.") for o in ops), (name, ops)
            pair = "float2" in params
            assert {o.rsplit(".", 1)[1] for o in ops} == ({"u64"} if pair else {"f32"}), (name, params, ops)
            seen.add(pair)
        assert seen == {True, False}, name


def test_no_weak_store_to_what_is_waited_for():
    text = open(SRC).read()
    kernels = text[text.index("k_fwdb_flow("):text.index("k_flowb_prep(")]
    stores = re.findall(r"\b(st[12]<V>|put_row(?:<V>)?)\(row_at\((\w+)", kernels)
    assert {to for how, to in stores if how.startswith("st")} <= {"gsp", "gtr"}   # outputs of the pass
    assert {to for how, to in stores if how.startswith("put")} == {"pqs", "tqs", "gs"}
