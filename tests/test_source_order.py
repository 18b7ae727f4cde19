"""Orders that the kernels' sources have to keep and that no run shows reliably: a load that happens to be slow
reads what a store ahead of it in program order has already replaced, or a cache line keeps what it held, once in
very many launches.

The row's length is read by every warp of the row's CTAs and replaced by the verification in the same launch.  The
store has to stand after the point that every reader has passed.

A grid may be resident while the kernel before it still writes the grid's inputs (programmatic launches), so none
of them is read through the non-coherent path, which asks for data that nothing writes while the grid runs.
"""
import os

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_20186_gb300", "csrc")


def _source(name: str) -> str:
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _positions(text: str, what: str):
    at, out = text.find(what), []
    while at >= 0:
        out.append(at)
        at = text.find(what, at + 1)
    return out


# the kernel's source, the point every reader of the length has passed
@pytest.mark.parametrize("name,passed", [("rescan.cu", "mbar_wait_polls(&bars[3], 0, a.msg_wait_polls)"),
                                         ("index.cu", "__syncthreads();\n    const int32_t L = s_ver[1];")],
                         ids=["rescan", "index"])
def test_length_is_stored_after_every_read(name, passed):
    text = _source(name)
    reads, stores = _positions(text, "__ldcg(a.lens + b)"), _positions(text, "a.lens[b] = ")
    wait = _positions(text, passed)
    assert len(reads) == 1 and len(wait) == 1 and stores
    assert reads[0] < wait[0] < min(stores)


def test_no_load_through_the_non_coherent_path():
    for name in sorted(os.listdir(CSRC)):
        text = _source(name)
        for what in ("__ldg(", "ld.global.nc"):
            assert what not in text, (name, what)
