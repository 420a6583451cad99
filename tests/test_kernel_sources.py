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


def test_what_the_previous_kernel_may_write_is_not_read_as_read_only():
    """A kernel that starts while the previous one of its stream drains reads x, lists and their lengths behind
    griddepcontrol.wait.  A load that is declared read-only may be moved in front of it: these kernels have none but of weights."""
    waiting = [p for p in SOURCES if "griddepcontrol.wait" in code(p)]
    assert len(waiting) >= 6
    for path in waiting:
        text = code(path)
        assert "__ldg(" not in text, path
        kernels = re.split(r"__global__", text)[1:]
        for kernel in kernels:
            if "griddepcontrol.wait" not in kernel:
                continue
            read_only = re.findall(r"\bconst\s+\w+\s*\*\s*(?:const\s+)?__restrict__\s+(\w+)", kernel[:kernel.rindex("griddepcontrol.wait")])
            read_only += re.findall(r"\bconst\s+[\w\s]+\*\s*(?:const\s+)?__restrict__\s+(\w+)", kernel.split("static", 1)[0])
            assert set(read_only) <= {"codes", "meta", "records"}, (path, read_only)


def test_no_launch_has_less_shared_memory_than_the_kernel_may_assume():
    """A kernel that sees its shared memory as one object may have any part of it read early, behind a condition or not: what a
    launch can do without lies behind the object."""
    sizes = [(p, m) for p in SOURCES for m in re.findall(r"sizeof\(\w*Smem<[^()]*>\)[^;]*;", code(p))]
    assert len(sizes) >= 8
    for path, text in sizes:
        assert not re.search(r"sizeof\(\w*Smem<[^()]*>\)\s*-", text), (path, text)


def test_a_cta_whose_bounded_wait_ran_out_stays_until_the_others_have_sent():
    """The wait arrives at the cluster's barrier first, a late one is for that barrier and then for the data; a thread that sends
    waits afterwards or ends; and nobody takes an answer for granted."""
    helpers = code(os.path.join(ROOT, "paper_2511_04477_b200", "csrc", "spqt_gemv_device.cuh"))
    body = helpers[helpers.index("bool mbar_wait_cluster("):]
    body = body[:body.index("\n}")]
    assert re.search(r"cluster_sent\(\);.*while \(!mbar_try<true>.*> kWaitNs.*if \(late\) return false;.*barrier\.cluster\.wait.*late = true;", body, flags=re.S)
    for path in SOURCES:
        text = code(path)
        if not path.endswith(".cu") or "st_async_" not in text:
            continue
        sends = [m.start() for m in re.finditer(r"\bst_async_\w+\(", text)]
        waits = [m.start() for m in re.finditer(r"\bmbar_wait_cluster\(", text)]
        assert len(sends) == len(waits) == 1 and sends[0] < waits[0], path
        between = text[sends[0]:waits[0]]
        assert not re.search(r"__sync|cluster_wait\(", between), (path, "a wait for something else in between")
        assert re.search(r"[!=,(]\s*$", text[:waits[0]]), (path, "an answer that nobody looks at")
        behind = text[waits[0]:text.index("__global__", waits[0])] if "__global__" in text[waits[0]:] else text[waits[0]:]
        if "__syncthreads" in behind:    # those that do not wait for stores but go on
            assert re.search(r"if \(tid >= \w+\) \{\s*cluster_sent\(\);\s*\} else \{", between), path


def test_a_list_without_a_length_is_no_list():
    """The index collection leaves no length where totals were lost, and the products that take a list look for that."""
    csrc = os.path.join(ROOT, "paper_2511_04477_b200", "csrc")
    collect = code(os.path.join(csrc, "spqt_sparsify.cu"))
    assert re.search(r"if \(!there\) \*count = kListLost;.*\*count = all < kNone \? \(int\)all : kListLost;", collect, flags=re.S)
    assert collect.count("totals.exchange(") == len(re.findall(r"totals\.exchange\([^;]*, count\);", collect)) == 2
    for name in ("spqt_gemv.cu", "spqt_kquant.cu", "spqt_gemm_small.cu"):
        text = code(os.path.join(csrc, name))
        reads = len(re.findall(r"ld_global_u32\((?:a\.count|count_ptr)\)", text))
        assert reads >= 1 and len(re.findall(r"LIST && count < 0\b|not_a_number_if\(count < 0, ", text)) == reads, name


def test_hints_stay_within_buffers_whose_size_is_known():
    """A given list has as many entries as its length says, which is read behind the wait; hints are given before it."""
    for path in SOURCES:
        for what in re.findall(r"\bprefetch_l2\(([^,]*),", code(path)):
            assert "idx" not in what, (path, what)
