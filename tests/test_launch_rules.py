"""What the kernels must keep to because each is launched as a programmatic dependent of the one before it (and may be resident
while that one, or a caller's kernel, still runs): read from the sources, since a violation would be a race on the device."""
import re
import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_1805_11046_b200" / "csrc"


def _sources():
    out = {}
    for f in sorted(CSRC.glob("*.cu*")):
        out[f.name] = re.sub(r"//[^\n]*", "", f.read_text())
    return out


def _body(text, at):
    """The braces that open at or after `at`, with what is in them."""
    start = text.index("{", at)
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i + 1]
    raise AssertionError("unbalanced braces")


def _kernels():
    out = {}
    for name, text in _sources().items():
        for m in re.finditer(r"__global__[^;{]*?\bvoid\b[^;{]*?(\w+_kernel)\s*\(", text):
            i, depth = m.end(), 1                      # to the end of the parameter list (default arguments may hold braces)
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            out[m.group(1)] = _body(text, i)
    return out


EARLY = {"code_sums_kernel", "conv_terms_kernel"}        # the kernels that let their successor go at their start


def test_every_kernel_waits_for_the_one_before():
    kernels = _kernels()
    assert len(kernels) > 30
    for name, body in kernels.items():
        if name != "bounded_wait_selftest_kernel":       # (launched in the ordinary way)
            assert "pdl_wait()" in body, name
    assert {n for n, b in kernels.items() if "pdl_trigger()" in b} == EARLY
    for name in EARLY:
        assert "tmem_alloc" not in kernels[name]         # a successor could take the tensor memory it waits for


def test_what_an_early_kernel_writes_is_read_by_ordinary_loads():
    """Code sums and zero-point terms: their reader is resident while they are written, which the non-coherent path excludes."""
    sources, kernels = _sources(), _kernels()
    at = _body(sources["qbp_mma.cuh"], sources["qbp_mma.cuh"].index("long long at(int64_t i) const"))
    assert "load_after_wait(" in at and "__ldg" not in at
    assert "__ldg" not in kernels["conv_terms_kernel"]   # (reads the code sums of the launch before)
    for name in ("qbp_mma_kernel", "qbp_conv2_kernel", "qbp_mma2_kernel", "qbp_wgrad_kernel", "qbp_wgrad2_kernel"):
        for m in re.finditer(r"__ldg\(([^;]*);", kernels[name]):
            assert m.group(1).startswith("P.ep_fold"), (name, m.group(0))      # (written by bn_out_range_kernel)


def test_no_bounded_wait_starts_its_clock_before_the_kernel_may_work():
    """The waits on barriers give up after about a second.  Every role therefore waits for the kernels before this one, however
    long those run, ahead of the first barrier that only completes once copies have been issued.  (The producer's first waits are
    on stages that nothing has filled yet: they pass at once.)"""
    sources = {f.name: f.read_text() for f in CSRC.glob("*.cu")}
    seen = 0
    for name, text in sources.items():
        if "-- MMA issuer" not in text:
            continue
        issuer, epilogue = text.index("-- MMA issuer"), re.search(r"//\s-+ epilogue", text).start()
        assert issuer < epilogue, name
        waiting = r"mbar_wait|_mma_loop|mma_loop_|_dispatch"
        for role in (text[issuer:epilogue], text[epilogue:]):
            assert "pdl_wait();" in role, name
            assert role.index("pdl_wait();") < re.search(waiting, role).start(), name
        seen += 1
    assert seen == 5                                     # the products' files


def test_regions_to_clear_beyond_the_room_for_them_are_refused(tmp_path):
    """The record that travels with a launch by value: one region too many is an error of the call, and what lies behind stays."""
    src = tmp_path / "zero.cpp"
    src.write_text("""
        #include "qbp_common.cuh"
        #include <cstring>
        namespace qbp { int fail(int status, const char *, ...) { return status; } }
        struct Guarded { qbp::ZeroJobs z; unsigned char behind[256]; };
        int main()
        {
            Guarded g{};
            memset(g.behind, 7, sizeof g.behind);
            uint32_t word = 0;
            for (int i = 0; i < qbp::kMaxZeroJobs; ++i) if (g.z.add(&word, i + 1) != QBP_OK) return 1;
            if (g.z.add(&word, 0) != QBP_OK || g.z.count != qbp::kMaxZeroJobs) return 2;       // nothing to clear: no room needed
            if (g.z.add(&word, 1) == QBP_OK || g.z.count != qbp::kMaxZeroJobs) return 3;
            for (int i = 0; i < qbp::kMaxZeroJobs; ++i) if (g.z.p[i] != &word || g.z.words[i] != i + 1) return 4;
            for (unsigned char b : g.behind) if (b != 7) return 5;
            return 0;
        }""")
    subprocess.run(["g++", "-std=c++17", "-I", str(CSRC), "-I", "/usr/local/cuda/include", str(src), "-o", str(tmp_path / "zero")], check=True)
    assert subprocess.run([str(tmp_path / "zero")]).returncode == 0
