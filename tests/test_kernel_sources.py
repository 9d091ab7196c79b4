"""Properties of the kernel sources that no run on a healthy GPU can show."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37001_b200", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def test_a_cta_that_gave_up_merges_nothing():
    """Shared items: the merge takes its item and its rows' tokens from shared memory, which a CTA that gave up may never
    have written; addresses of out and lse would come from whatever was there before."""
    calls = re.findall(r"[^;{}]*\bmerge_cluster\s*\(\s*prm\b[^;]*;", _source("psa_attn_sm100.cu"))
    assert len(calls) == 1
    assert re.search(r"if\s*\([^;]*\*abort_flag\s*==\s*0[^;]*\)\s*merge_cluster", calls[0]), calls[0]


def _definitions(name):
    """Names of the functions and types that a source file defines outside functions, types and unnamed namespaces."""
    text, found, i = _source(name), [], 0
    text = re.sub(r'extern\s+"C"\s*\{|namespace\s+\w+\s*\{', lambda m: " " * len(m.group()), text)   # (looked through)
    head = 0
    while i < len(text):
        if text[i] == "{":
            intro, depth = text[head:i], 1
            while depth:
                i += 1
                depth += {"{": 1, "}": -1}.get(text[i], 0)
            m = re.search(r"\bstruct\s+(\w+)\s*$", intro) or re.search(r"\b(\w+)\s*\((?:[^()]|\([^()]*\))*\)\s*(?:const)?\s*$", intro)
            if m and "namespace" not in intro and not re.search(r"\bstatic\b", intro):
                found.append(m.group(1))
            head = i + 1
        elif text[i] in ";}":
            head = i + 1
        i += 1
    return found


def test_no_two_files_define_the_same_name():
    """One library: two inline functions or types of one name in one namespace are one to the linker."""
    where = {}
    for f in sorted(os.listdir(CSRC)):
        for name in _definitions(f):
            where.setdefault(name, set()).add(f)
    assert {"attn_fwd_kernel", "launch_mask_build", "make_geom", "Geom", "psa_attn_fwd", "axis_set"} - set(where) == {"make_geom"}
    assert {n: fs for n, fs in where.items() if len(fs) > 1} == {}
