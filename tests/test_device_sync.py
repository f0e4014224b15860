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
