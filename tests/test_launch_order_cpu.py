"""Order of the programmatic-launch calls in the kernels, checked on the sources (a race between kernels cannot be shown
by running them): a kernel lets its dependents go only behind its own wait, so that what a successor reads ahead of ITS
wait cannot still be in the making two kernels further up."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_17803_b200", "csrc")
# They stand directly behind a kernel of the same call that keeps the rule (the scorer, the selection), or are an ordinary
# launch that nothing precedes.
TRIGGER_FIRST = {"topk_regs_kernel", "topk_smem_kernel", "topk_generic_kernel", "expand_clusters_kernel", "fetch_kernel"}


def kernels():
    """(name, text) of every kernel, and of the resolution body that two of them share."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        heads = list(re.finditer(r"__global__[^{;]*?\b(\w+)\s*\(\s*(?:Geometry|const|ResolveArgs|ClusterArgs|uint|int|float)|"
                                 r"void (resolve_body)\(", text))
        for m, end in zip(heads, [h.start() for h in heads[1:]] + [len(text)]):
            yield m.group(1) or m.group(2), text[m.start():end]


def test_dependents_are_released_behind_the_wait():
    seen = set()
    for name, text in kernels():
        seen.add(name)
        trigger, wait = text.find("pdl_launch_dependents()"), text.find("pdl_wait()")
        if trigger >= 0 and name not in TRIGGER_FIRST:
            assert 0 <= wait < trigger, name
    assert TRIGGER_FIRST <= seen
    assert {"page_score_kernel", "page_score_mma_kernel", "attn_kernel", "gather_kernel", "summaries_kernel", "medoid_rows_kernel",
            "admit_kernel", "resolve_body"} <= seen
