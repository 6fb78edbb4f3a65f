"""Rules of the CUDA sources that no run can show to be kept: what they guard against depends on how
the compiler places an instruction, or on two SMs' timing."""

import os
import re

from paper_2606_07116_gb300 import build as B


def source(name):
    """A source file without its comments."""
    with open(os.path.join(B.CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def block(text, start):
    """The braced block that begins at or after `start`."""
    a = text.index("{", start)
    depth = 0
    for i in range(a, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[a:i + 1]
    raise AssertionError("unbalanced braces")


def test_mx_gemm_commits_its_teardown_barrier_only_after_an_abort():
    """An arrival that nobody waits for may reach a CTA that has ended: the commit to `done` belongs to the
    abort's teardown, goes to the issuer's own CTA, and is waited for there."""
    text = source("gemm_mx.cu")
    commits = re.findall(r"mma2_commit\w*\(done\)", text)
    assert commits == ["mma2_commit(done)"]
    teardown = block(text, text.index("if (*abort) {"))
    assert teardown.index("mma2_commit(done)") < teardown.index("wait_teardown(done, 0)")


def test_waits_for_tensor_memory_loads_name_their_registers():
    """A tcgen05.wait::ld that does not list the loaded registers orders memory accesses only: the compiler may
    move or spill them before their data is there. Each wait is in the load's own statement or takes them as
    operands."""
    for name in sorted(os.listdir(B.CSRC)):
        text = source(name)
        for m in re.finditer(r"tcgen05\.wait::ld", text):
            statement = text[text.rindex("asm volatile(", 0, m.start()):text.index(";\n}", m.end())]
            assert "tcgen05.ld." in statement or '"+r"(' in statement, (name, statement)


def test_loops_over_tensor_memory_columns_keep_the_warp_together():
    """The .sync.aligned TMEM loads need all lanes of the warp at once. In a loop that issues them, lanes without a
    row or a channel to write take no `continue`, and the warp meets again before the next load."""
    for name in sorted(os.listdir(B.CSRC)):
        text = source(name)
        loops = [(m.start(), block(text, text.index(")", m.end()))) for m in re.finditer(r"\bfor \(", text)
                 if re.match(r"for \([^{};]*;[^{};]*;[^{}]*?\) \{", text[m.start():])]
        for start, body in loops:
            inner = [b for _, b in loops if b in body and b != body]
            own = body
            for b in inner:
                own = own.replace(b, "")
            if not re.search(r"\btmem_ld_\w+\(", own):
                continue
            assert "continue;" not in own, (name, own[:200])
            if "store_out<" in own or "p.out)" in own:
                assert re.search(r"__syncwarp\(\)|__all_sync\(", own), (name, own[:200])


def test_few_token_gemm_reads_early_only_what_its_contract_names():
    """Before the wait for the kernel ahead the few-token GEMM may read the weights (codes, scales, row sums) only
    in the EARLY instantiation (offq.h names those calls), else only prefetch them, and touches nothing else of
    its inputs."""
    text = source("gemm_few.cu")
    body = block(text, text.index("w4a4_few_kernel(const FewParams p)"))
    for f, reads in (("first_w", "load_w("), ("constants", "p.w_scale")):
        own = block(body, body.index(f"auto {f} = [&]"))
        assert reads in own
        body = body.replace(own, "")
    load = body[body.index("auto load_w = "):]
    body = body.replace(block(load, 0), "")
    start = body.index("if constexpr (EARLY) {")
    early = block(body, start)
    late = block(body, start + len("if constexpr (EARLY) ") + len(early))
    assert early.index("first_w();") < early.index("griddep_wait();") > early.index("constants();")
    before, after = late.split("griddep_wait();")
    assert "first_w();" in after and not re.search(r"first_w\(\)|constants\(\)|__ldg|cp_async|p\.a_|p\.out", before)
    assert before.count(";") == 1 and "prefetch_w();" in before
    head = body[:start]
    assert not re.search(r"first_w\(\)|constants\(\)|__ldg|cp_async<|p\.(a_\w+|out|w_scale|rowsum)\b", head)
    assert re.search(r"return T <= kEarlyTokens && ", text)


def test_kernels_that_finish_weight_tables_do_not_release_their_dependents_early():
    """At up to 4 tokens offq_w4a4_linear reads codes, scales and row sums before its wait."""
    for name, kernel in (("quant.cu", "weight_repack_kernel("), ("quant_group.cu", "weight_group_sums_kernel(")):
        text = source(name)
        body = block(text, text.index(kernel))
        assert "griddep_wait();" in body and "griddep_launch_dependents" not in body, kernel


def test_the_host_keeps_no_plain_mutable_statics():
    """The ABI's calls may come from several threads at once: what the host code keeps between calls is atomic,
    under a mutex or set once."""
    for name in sorted(os.listdir(B.CSRC)):
        text = source(name)
        for m in re.finditer(r"^\s+static (?!constexpr|const |_?_?device|__forceinline__|inline|_assert)([^;(]*?)[;={]", text,
                             flags=re.M):
            decl = m.group(1)
            var = decl.split()[-1]
            synchronised = (re.search(r"std::(atomic|mutex|once_flag)", decl) or f"__atomic_load_n(&{var}" in text
                            or "std::call_once(once" in text and "std::once_flag once;" in text[m.end():m.end() + 60])
            assert synchronised, (name, decl)
    assert sum(source(n).count("cudaDevAttrMultiProcessorCount") for n in os.listdir(B.CSRC)) == 1
