"""Barriers of the CTA-pair kernel that the other CTA arrives on: arrivals and waits name cluster scope. Between two CTAs a release or
an acquire at CTA scope orders nothing, and the tensor core then reads the other CTA's shared memory unordered with its stores;
a run cannot be relied on to show that, so the sources are looked at."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2609_22755_b200" / "csrc"


def test_remote_arrivals_name_cluster_scope():
    forms = [f for p in CSRC.glob("*.cu*") for f in re.findall(r"mbarrier\.arrive[\w.:]*", p.read_text()) if "shared::cluster" in f]
    assert forms and all(re.match(r"mbarrier\.arrive\.(relaxed|release)\.cluster\.", f) for f in forms), forms


def test_waits_behind_the_other_cta_name_cluster_scope():
    text = (CSRC / "nsp_bwd_pair.cu").read_text()
    # arrived on by the other CTA's threads, or counting the bytes of its loads
    remote = set(re.findall(r"arrive_lead\(&s\.(\w+)\)", text)) | set(re.findall(r"lead \+ off\(&s\.(\w+)\)", text))
    remote |= set(re.findall(r"load_(?:row|col)\([^;]*?&s\.(\w+)", text))
    assert {"bar_p_ready", "bar_ds_ready", "bar_s_read", "bar_dq_empty", "bar_x_peer", "bar_kv", "bar_qr_full"} <= remote
    for name in remote:
        waits = [w for w in re.findall(r"(\w*wait\w*)\(([^;{}]*)", text) if re.search(r"&s\.%s\b" % name, w[1])]
        assert waits and all(w[0].startswith("cluster_") for w in waits), (name, waits)


def test_shared_memory_is_not_handed_over_by_the_relaxed_arrival():
    # dS^T in shared memory: a barrier of the CTA that wrote it, then one released arrival for all of it
    text = (CSRC / "nsp_bwd_pair.cu").read_text()
    assert not re.search(r"arrive_lead\(&s\.bar_x_\w+\)", text)
    assert re.search(r"cluster_arrive_release\(lead \+ off\(&s\.bar_x_peer\)\)", text)
