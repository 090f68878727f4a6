"""Kernels launched before the one in front of them has ended (launch_next):
each waits in its first statement, and what the kernel just before writes is
never read through the read-only path, nor by assembly that the compiler may
move. Checked on the sources: a compiler that happens to keep the order would
hide a breach from any run."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_15876_gb300", "csrc")
SOURCE = {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu*"))}

# kernel -> its arguments that the kernel launched just before it writes (read
# as well as added to; arguments only added to with atomics need nothing)
WRITTEN_JUST_BEFORE = {
    "k_block_sums": ["in"], "k_scan_sums": ["sums"], "k_scan_tiles": ["in", "sums"],
    "k_pix_scatter": [], "k_pix_commit": ["bk"], "k_pix_finish": ["state1", "bk"],
    "k_fifo_append": ["rank"], "k_fifo_advance": [],
    "k_place_queues": ["flist"], "k_place_fifo": ["flist"],
    "k_filter": ["fconst"], "k_bwd_record": ["adj"], "k_bwd_params": ["part"],
}


def _kernel(name):
    for text in SOURCE.values():
        m = re.search(r"__global__ void[^;{]*?\b%s\(([^{]*)\)\s*\{(.*?)\n\}" % name, text, re.S)
        if m:
            return m.group(1), m.group(2)
    raise AssertionError(f"kernel {name} not found")


def test_every_overlapped_kernel_is_listed_and_waits_first():
    launched = set()
    for text in SOURCE.values():
        launched |= set(re.findall(r"launch_next\((k_\w+)", text))
    assert launched == set(WRITTEN_JUST_BEFORE)
    for name in launched:
        _, body = _kernel(name)
        assert body.lstrip().startswith("grid_order();"), name


def test_what_the_kernel_before_writes_is_read_with_ordinary_loads():
    for name, fresh in WRITTEN_JUST_BEFORE.items():
        args, body = _kernel(name)
        for arg in fresh:
            decl = next(a for a in args.split(",") if re.search(r"\b%s$" % arg, a.strip()))
            assert "__restrict__" not in decl, (name, decl)
            assert not re.search(r"__ldg\(\s*(&|reinterpret_cast<[^>]*>\()?\s*%s\b" % arg, body), (name, arg)
    # read in functions that kernels share
    assert not re.search(r"__ldg\(\s*&?(bk\.r|adj\.[kg]|ridx)\b", "".join(SOURCE.values()))
    text = SOURCE["k_filter.cu"]
    assert "Fresh<float4> k;" in text and "Fresh<float2> g;" in text
    assert "__ldg" not in re.search(r"float4 load_const\((.*?)\n}", text, re.S).group(1)


def test_loads_in_assembly_stay_behind_the_wait():
    for file, text in SOURCE.items():
        for m in re.finditer(r'asm( volatile)?\("ld\.global\.(?!nc)(.*?);\n', text, re.S):
            assert m.group(1) and '"memory"' in m.group(2), (file, m.group(0)[:60])
