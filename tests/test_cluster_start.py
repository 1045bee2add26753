"""Another CTA's shared memory may be accessed only once that CTA has started,
which a cluster barrier is there to guarantee. Reads the kernels' source: in
the body of every kernel, a cluster barrier stands ahead of the first access to
a shared::cluster address of another CTA (stores, loads, arrivals, TMA and MMA
completions on a peer's barrier)."""

import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2606_04945_gb300" / "csrc"
BARRIER = re.compile(r"\bcluster_(sync|started_wait)\s*\(|barrier\.cluster\.wait")
REMOTE = re.compile(r"\b(st|ld)_shared_cluster\w*\s*\(|\b(st|ld|atom|red)\.[\w.]*shared::cluster|"
                    r"\bmbar_arrive_cluster\w*\s*\(|\btma_load_2d_pair\s*\(|\btc_commit_pair_multicast\s*\(|"
                    r"\bmma_\w+_pair\s*\(")


def strip_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def kernels(text):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\b", text):
        head = text[m.end():text.index("{", m.end())]
        names = [n for n in re.findall(r"(\w+)\s*\(", head) if n != "__launch_bounds__"]
        start = text.index("{", m.end())
        depth, i = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
            if depth == 0:
                break
        yield names[0], text[start:i]


def first(pattern, text):
    m = pattern.search(text)
    return m.start() if m else None


def unguarded(body):
    remote, barrier = first(REMOTE, body), first(BARRIER, body)
    return remote is not None and (barrier is None or barrier > remote)


SOURCES = sorted(CSRC.glob("*.cu"))


@pytest.mark.parametrize("path", SOURCES, ids=lambda p: p.name)
def test_barrier_before_first_remote_access(path):
    for name, body in kernels(strip_comments(path.read_text())):
        assert not unguarded(body), f"{path.name}: {name} reaches into another CTA before any cluster barrier"


def test_finds_the_kernels_with_remote_accesses():
    found = {name for p in SOURCES for name, body in kernels(strip_comments(p.read_text())) if REMOTE.search(body)}
    assert {"sgat_quant_rows_kernel", "attn_vquant_kernel", "w4a4_gemm_few_kernel", "w4a4_gemm_tma_pair_kernel"} <= found
    assert unguarded("{ st_shared_cluster_f32(mapa_shared(p, r), v); cluster_sync(); }")
