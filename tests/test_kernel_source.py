"""Rules of the memory model that the kernels' sources have to keep and that no run can be relied on to show: a program
without the scope or the wait that the model asks for gives right results as long as the hardware is kinder than it."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2602_07711_gb300" / "csrc"
SOURCES = {p.name: re.sub(r"//.*", "", p.read_text()) for p in sorted(CSRC.iterdir()) if p.suffix in (".cu", ".cuh")}


def body(text, name):
    """The text of the function `name` from its parameter list to its closing brace in the first column."""
    start = text.index(name + "(")
    return text[start:text.index("\n}\n", start)]


def test_arrivals_on_another_ctas_barrier_are_of_cluster_scope():
    seen = 0
    for name, text in SOURCES.items():
        for op in re.findall(r"mbarrier\.arrive[\w.:]*shared::cluster[\w.:]*", text):
            assert re.search(r"\.(release|relaxed)\.cluster\.", op), (name, op)
            seen += 1
    assert seen


def test_waits_of_the_pair_kernel_acquire_at_cluster_scope():
    text = SOURCES["gemm_tc.cu"]
    for name in ("pair_pass_kernel", "settle_loads"):
        assert not re.search(r"\bmbar_wait\(", body(text, name)), name
    assert "try_wait.parity.acquire.cluster." in body(text, "mbar_wait_cluster")


def test_values_of_the_chains_other_kernels_are_not_read_ahead_of_the_wait():
    """A kernel that may start before its predecessor ends reads what that one writes after grid_wait() alone: no
    __restrict__ on the pointer, no plain load through it."""
    for name, text in SOURCES.items():
        assert not re.search(r"double\*\s+__restrict__\s+(h16d|alpha_dev2)\b", text), name
        for kernel in re.findall(r"__global__[^;{]*?\b(\w+_kernel)\(", text):
            code = body(text, kernel)
            if "grid_wait()" in code:
                assert not re.search(r"\b(h16d|alpha_dev2)\[[^\]]*\](?!\s*=[^=])", code), (name, kernel)
