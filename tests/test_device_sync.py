"""Rules of the kernels' synchronisation that hold by the text of the sources alone
(CPU): a breach shows on the GPU only now and then, or never."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_15478_gb300", "csrc")


def sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(f) as h:
            out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", h.read())
    assert len(out) > 10
    return out


def test_hand_backs_release():
    """An arrival hands memory over, so it has to be a release (the default)."""
    for name, text in sources().items():
        assert not re.search(r"mbarrier\.arrive[\w.:]*\.relaxed", text), name


def bodies(text):
    """The text of every kernel, from its name to its closing brace."""
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\([^{;]*\)\s*\{", text):
        depth, k = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), text[m.end():k]


def test_clusters_meet_before_remote_accesses():
    """Another CTA's shared memory may be accessed once that CTA is known to run: a
    kernel with such accesses has a barrier of the cluster in front of the first."""
    remote = re.compile(r"\b(map_rank|ld_cluster_\w+|st_cluster_\w+|st_async_\w+|"
                        r"mbar_arrive_remote\w*|run_link_\w+)\b")
    found = []
    for name, text in sources().items():
        for kernel, body in bodies(text):
            first = remote.search(body)
            if not first:
                continue
            found.append(kernel)
            barrier = body.find("cluster_sync_all()")
            assert 0 <= barrier < first.start(), (name, kernel)
    assert sorted(found) == ["k_dp_split", "k_seg_cluster"]
