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
