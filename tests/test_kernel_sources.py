"""Rules of the memory model that the kernels' sources have to keep.  What breaks one of them need not show in a result, and
may not be tried on a GPU, so the text of the sources is what is looked at."""
import glob
import os
import re

from conftest import ROOT

SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2511_04477_b200", "csrc", "*.cu*")))


def code(path):
    """The source without comments."""
    text = open(path).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_waits_for_stores_of_other_ctas_acquire_at_cluster_scope():
    """mbarrier.try_wait acquires at the scope of the CTA unless it says otherwise; data that other CTAs of a cluster sent with
    st.async need the cluster's."""
    senders = [p for p in SOURCES if p.endswith(".cu") and "st_async_" in code(p)]
    assert len(senders) >= 4
    for path in senders:
        waits = re.findall(r"\bmbar_wait\w*\(", code(path))
        assert waits and set(waits) == {"mbar_wait_cluster("}, (path, waits)
    helpers = open(os.path.join(ROOT, "paper_2511_04477_b200", "csrc", "spqt_gemv_device.cuh")).read()
    forms = re.findall(r"mbarrier\.try_wait\.[a-z0-9_.:]*", helpers)
    assert sorted(forms) == ["mbarrier.try_wait.parity.acquire.%s.shared::cta.b64" % s for s in ("cluster", "cta")]
