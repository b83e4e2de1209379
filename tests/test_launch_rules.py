"""What the kernels must keep to because each is launched as a programmatic dependent of the one before it (and may be resident
while that one, or a caller's kernel, still runs): read from the sources, since a violation would be a race on the device."""
import re
import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_1805_11046_b200" / "csrc"


def _sources(comments=False):
    out = {}
    for f in sorted(CSRC.glob("*.cu*")):
        text = f.read_text()
        out[f.name] = text if comments else re.sub(r"//[^\n]*", "", text)
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


def _kernels(comments=False):
    out = {}
    for name, text in _sources(comments).items():
        for m in re.finditer(r"__global__[^;{]*?\bvoid\b[^;{]*?(\w+_kernel)\s*\(", text):
            i, depth = m.end(), 1                      # to the end of the parameter list (default arguments may hold braces)
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            out[m.group(1)] = _body(text, i)
    return out


EARLY = {"code_sums_kernel", "conv_terms_kernel"}        # the kernels that let their successor go before they end
PRODUCTS = {"qbp_mma_kernel", "qbp_mma2_kernel", "qbp_conv2_kernel", "qbp_conv2t_kernel", "qbp_wgrad_kernel", "qbp_wgrad2_kernel"}


def test_every_kernel_waits_for_the_one_before():
    kernels = _kernels()
    assert len(kernels) > 30
    for name, body in kernels.items():
        if name != "bounded_wait_selftest_kernel":       # (launched in the ordinary way)
            assert "pdl_wait()" in body, name
    assert {n for n, b in kernels.items() if "pdl_trigger()" in b} == EARLY
    for name in EARLY:
        assert "tmem_alloc" not in kernels[name]         # a successor could take the tensor memory it waits for


def test_a_successor_that_does_not_wait_starts_behind_the_wait_of_the_kernel_before_it():
    """A product told that its launch follows its sums or terms (`beside`) reads its operands without a wait of its own: the kernel
    that makes them may let it go only once everything before is complete.  Without that, letting go ahead of the wait is allowed:
    the successor waits itself."""
    kernels, sources = _kernels(), _sources()
    steps = lambda name: re.findall(r"(if \([^;]*?\) )?(pdl_trigger|pdl_wait)\(\)", kernels[name])
    assert steps("conv_terms_kernel") == [("", "pdl_wait"), ("", "pdl_trigger")]
    assert steps("code_sums_kernel") == [("if (!BESIDE) ", "pdl_trigger"), ("", "pdl_wait"), ("if (BESIDE) ", "pdl_trigger")]
    # who tells it: the launch of the sums, with the kernel's own form, and the launch of the terms, right behind which the product comes
    quant, mma = sources["qbp_quant.cu"], sources["qbp_mma.cu"]
    assert quant.count("*beside = ahead") == 1 and quant.count("*beside =") == 2
    assert "if (ahead) launch(code_sums_kernel<true>," in quant and "else       launch(code_sums_kernel<false>," in quant
    assert len(re.findall(r"\bbeside = true", mma)) == 1
    assert "launch" not in re.sub(r"QBP_LAUNCH_OK", "", mma[mma.index("launch(conv_terms_kernel,") + 6:mma.index("beside = true")])


def test_what_an_early_kernel_writes_is_read_by_ordinary_loads():
    """Code sums and zero-point terms: their reader is resident while they are written, which the non-coherent path excludes."""
    sources, kernels = _sources(), _kernels()
    at = _body(sources["qbp_mma.cuh"], sources["qbp_mma.cuh"].index("long long at(int64_t i) const"))
    assert "load_after_wait(" in at and "__ldg" not in at
    assert "__ldg" not in kernels["conv_terms_kernel"]   # (reads the code sums of the launch before)
    assert PRODUCTS <= {n for n, b in kernels.items() if "load_after_wait(" in b or ".at(" in b}
    for name in PRODUCTS:
        for m in re.finditer(r"__ldg\(([^;]*);", kernels[name]):
            assert m.group(1).startswith("P.ep_fold"), (name, m.group(0))      # (written by bn_out_range_kernel)


def _roles(name, body):
    """A product's kernel (with its comments): what comes before the MMA issuer, the issuer, the epilogue, what ends the kernel."""
    assert body.count("-- MMA issuer") == 1, name
    issuer, epilogue = body.index("-- MMA issuer"), [m.start() for m in re.finditer(r"//\s-+ epilogue", body)]
    end = body.rindex("if (timed_out) {")
    assert len(epilogue) == 1 and issuer < epilogue[0] < end, name
    cut = lambda a, b: re.sub(r"//[^\n]*", "", body[a:b])
    return cut(0, issuer), cut(issuer, epilogue[0]), cut(epilogue[0], end), cut(end, len(body))


def test_no_bounded_wait_starts_its_clock_before_the_kernel_may_work():
    """The waits on barriers give up after about a second.  Every role therefore waits for the kernels before this one, however
    long those run, ahead of the first barrier that only completes once copies have been issued; the issuer of a product that runs
    beside its sums need not, since its copies do not wait either.  (The producer's first waits are on stages that nothing has filled
    yet: they pass at once.)"""
    kernels = _kernels(comments=True)
    assert {n for n, b in kernels.items() if "-- MMA issuer" in b} == PRODUCTS
    waiting = r"mbar_wait|_mma_loop|mma_loop_|_dispatch"
    for name in PRODUCTS:
        before, issuer, epilogue, _ = _roles(name, kernels[name])
        guard, = re.findall(r"(if \([^;]*\) )?pdl_wait\(\);", issuer)
        assert guard in ("", "if (!P.beside) "), name
        assert issuer.index("pdl_wait();") < re.search(waiting, issuer).start(), name
        assert epilogue.index("pdl_wait();") < re.search(waiting, epilogue).start(), name
        # (the roles that copy operands or read their parameters, under the same condition, at their first use)
        working = [r for r in re.split(r"(?m)^    (?:\} else )?if \(warp", before)[1:] if re.search(r"tma_load|P\.qa->", r)]
        assert working and all("pdl_wait();" in r for r in working), name
        assert bool(guard) == all("P.beside" in r for r in working), name


def test_a_product_beside_its_sums_waits_before_it_reads_them_or_writes():
    """Its epilogue, unconditionally and first; nothing else reads sums or terms, or writes; the status word, which the launch before
    may clear, is raised behind a wait as well."""
    kernels, seen = _kernels(comments=True), 0
    touching = r"load_after_wait\(|\.at\(|rowterm|colterm|tot_g|acc_out|P\.out\b|P\.dW|P\.mapC|st_sum|tma_store|st\.global|raise_timeout|atomicAdd"
    for name in sorted(PRODUCTS):
        before, issuer, epilogue, end = _roles(name, kernels[name])
        wait = re.search(r"(?m)^\s*pdl_wait\(\);", epilogue)
        assert wait and "{" not in re.sub(r"\{[^{}]*\}", "", epilogue[:wait.start()]), name      # (not inside a branch of the role)
        assert not re.search(touching, epilogue[:wait.start()]), name
        if "P.beside" not in kernels[name]:
            continue
        seen += 1
        for role in (re.sub(r"(if \([^;]*\) )?tma_prefetch_desc\([^;]*;", "", before), issuer):
            assert not re.search(touching, role), (name, re.search(touching, role).group(0))
        raised = end.index("raise_timeout(")
        assert re.search(r"(?m)^\s*pdl_wait\(\);", end[:raised]), name
    assert seen == 5


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
