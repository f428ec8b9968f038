"""Memory scopes of the wavefront kernels, read from their sources: a shared
word that another CTA of the cluster stores to while this one runs has a
type of its own and is only loaded at cluster scope (a CTA-scope load does not
pair with a store from outside the CTA)."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2506_21932_gb300" / "csrc"


@pytest.mark.parametrize("name", ["trisolve.cuh", "k_btri.cu"])
def test_words_that_a_peer_counts_in_are_read_at_cluster_scope(name):
    src = (CSRC / name).read_text()
    # addresses of a neighbour's words that are kept for the length of a tile
    words = set(re.findall(r"unsigned \w+ = [^;]*peer_addr\(&sh\.(\w+)", src))
    assert words == {"taken"}
    assert re.search(r"\bPeerCounter taken\b", src)
    assert not re.search(r"ld_acq_cta\([^)]*taken", src)
    # the pointer that may hold its address is read at cluster scope only
    pointers = set(re.findall(r"int\* (\w+) = [^;]*&sh\.taken[^;]*\.v;", src))
    assert pointers == {"word"}
    assert set(re.findall(r"(\w+)\(word\)", src)) == {"ld_acq_cluster"}
    load = re.search(r"int ld_acq_cluster\(.*?\n\}", (CSRC / "mailbox.cuh").read_text(), re.S).group(0)
    assert re.findall(r"\bld\.[\w.:]+", load) == ["ld.acquire.cluster.shared::cta.s32"]
