"""Rules that the CUDA sources keep because breaking them shows on a GPU only by chance."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_14363_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def _block(text, start):
    """text from the first brace at or after `start` to the one that closes it."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def _kernels(text):
    """(head, body) of every kernel: its signature and its definition."""
    for m in re.finditer(r"__global__", text):
        body = _block(text, text.index(")", m.start()))
        yield text[m.start():text.index(body, m.start())], body


# Kernels whose predecessor is always a kernel of the same call that lets its dependents start after its own wait.
BEHIND_A_WAIT = {"project_reduce_kernel"}


@pytest.mark.parametrize("name", SOURCES)
def test_a_kernel_waits_before_it_lets_dependents_start(name):
    """Else a kernel that reads something before its own wait (weights, sequence lengths) could run beside one that was
    enqueued two calls before it and still writes that."""
    for head, body in _kernels(_code(name)):
        if "griddep_launch_dependents" in body:
            assert "griddep_wait" in body, head
            if any(k in head for k in BEHIND_A_WAIT):
                continue
            assert body.rindex("griddep_wait") < body.index("griddep_launch_dependents"), head


@pytest.mark.parametrize("name", SOURCES)
def test_what_another_grid_may_still_write_is_not_read_as_read_only(name):
    """A kernel that may start beside its producer reads with plain or .cg loads: the read-only path (__ldg, or what the compiler
    makes of a const __restrict__ pointer) is for data nobody writes during the whole life of the kernel, and the wait does
    not order it."""
    text = _code(name)
    assert "__ldg(" not in text
    for head, body in _kernels(text):
        if "griddep_wait" in body:
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", head), head


def test_a_product_that_quantizes_its_rows_reads_no_weight_before_its_wait():
    """The kernel before it is the caller's (resq_pack_weights, say), not a quantizer of the same call, and the option that a caller sets
    for resq_mixed_gemm promises nothing about it."""
    text = _code("decode_stream.cu")
    assert re.findall(r"\bp\.early_weights = ([^;]*)", text) == ["X ? 0 : g_early_weights ? g_early_weights : after_quantizer ? kAfterQuantizer : 0"]
    kernel = next(body for head, body in _kernels(text) if "mixed_gemm_stream_kernel" in head)
    assert kernel.index("if (!p.early_weights) griddep_wait();") < kernel.index("issue(0)")


def test_waits_are_bounded_by_the_library_s_limit():
    """Both forms of a bounded wait compare the clock with the limit that the caller may set.  Elsewhere it bounds only what a kernel does after a
    wait has run out: up to a tenth of a second for copies still in flight."""
    for name in SOURCES:
        if name != "ptx.cuh":
            text = _code(name)
            drains = re.findall(r"global_timer_ns\(\) - \w+ < (\d+)ull\) \{\}", text)
            assert text.count("global_timer_ns") == text.count("= global_timer_ns();") + len(drains), name
            assert all(int(ns) <= 100_000_000 for ns in drains), name
    text = _code("ptx.cuh")
    forms = [_block(text, m.start()) for m in re.finditer(r"\bbool mbar_wait\w*\(", text)]
    assert len(forms) == 2 and text.count("global_timer_ns") == 1 + sum(f.count("global_timer_ns") for f in forms)
    for f in forms:
        assert "const volatile unsigned long long*>(status + 2)" in f


TMEM_ACCESS = r"(?<!__forceinline__ void )\btmem_(?:ld|st)\d\w*\("
TMEM_ACCESSES = {"kv_prefill.cu": 7, "mixed_gemm.cu": 2, "mixed_gemm_mid.cu": 3, "project.cu": 2}


@pytest.mark.parametrize("name", SOURCES)
def test_a_tensor_memory_load_and_its_wait_are_one_statement(name):
    """Registers of a load on its way may be written at any time: between it and a wait of its own the compiler could move one."""
    text = _code(name)
    for m in re.finditer(r"\basm (?:volatile)?\(", text):
        end, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[end], 0)
            end += 1
        statement = text[m.start():end]
        assert ("tcgen05.ld." in statement) == ("tcgen05.wait::ld" in statement), (name, statement[:80])


@pytest.mark.parametrize("name", SOURCES)
def test_tensor_memory_is_reached_by_whole_warps(name):
    """A TMEM load or store is for all 32 lanes at once.  A loop in which lanes may part ways (rows, columns or outputs that some
    lanes do not have) brings them together again before the next iteration's access, and no lane goes on past a wait that
    ran out for another."""
    text = _code(name)
    found = list(re.finditer(TMEM_ACCESS, text))
    assert len(found) >= TMEM_ACCESSES.get(name, 0)  # a new name of the wrappers does not empty the rule
    for m in found:
        loops = [f for f in re.finditer(r"\bfor \(", text[:m.start()])]
        enclosing = None
        for f in loops:
            close, depth = f.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(text[close], 0)
                close += 1
            if text[close:].lstrip().startswith("{"):
                body = _block(text, close)
                if text.index(body, close) + len(body) > m.start():
                    enclosing = (text.index(body, close), body)
        if enclosing is None:
            continue
        at, body = enclosing
        if re.search(r"\bcontinue;|\b\w+_ok\b", body[m.start() - at:]):
            assert "__syncwarp();" in body[:m.start() - at], (name, text[m.start():m.start() + 60])
    for m in re.finditer(r"if \(!mbar_wait\(&sh->acc_full", text):
        raise AssertionError((name, text[m.start():m.start() + 80]))


def test_warps_that_meet_at_a_barrier_leave_together():
    """The softmax warps that share rows of the prefill kernel meet at a named barrier, which has no time limit.  A wait that runs out in
    one of them is voted on at every such barrier and the outcome acted on, so that none goes on to a barrier where the others
    will not come."""
    text = _code("kv_prefill.cu")
    kernel = next(body for head, body in _kernels(text) if "attention_prefill_kernel" in head)
    votes = re.findall(r"([^;{}]*)\bgroup_any<32 \* WAYS>\(group, ([^;]*)", kernel)
    assert len(votes) == 3
    for before, predicate in votes:
        assert "!ok" in predicate and "(void)" not in before and re.search(r"\bif \($|= $", before), (before, predicate)


def test_scores_go_over_weights_only_behind_the_product_that_reads_them():
    """The weights of an output product lie in TMEM where later scores go.  Products are ordered by their issue only if they share
    accumulator and shape, which these two do not.  So the scores are issued behind a wait for the other's completion, or
    into the buffer of their stage, whose keys are awaited: expansion fills a stage only after the product that read it has freed it."""
    text = _code("kv_prefill.cu")
    kernel = next(body for head, body in _kernels(text) if "attention_prefill_kernel" in head)
    pair_at = kernel.index("if constexpr (PAIR)", kernel.index("int out_stage"))
    pair = _block(kernel, pair_at)
    one = _block(kernel, kernel.index("else", pair_at + len(pair)))
    loop = _block(pair, pair.index("for (int n = 0"))
    between = loop[loop.index("output_product("):loop.index("score_product(")]
    assert between.index("tc_commit_if(leader, &sh->pv_done[t])") < between.index("wait(&sh->pv_done[t], n & 1)"), between
    scores = _block(one, one.index("auto scores"))
    assert scores.index("!keys_ready()) return;") < scores.index("score_product(") and "stage, stage, N & 1)" in scores
    assert "output_product(out_stage, N & 1," in one and "tc_commit_if(leader, &sh->kv_empty[out_stage])" in one
    expand = kernel[kernel.index("for (; N < total_steps; ++N)"):kernel.index("expand_step<D>")]
    assert "mbar_wait(&sh->kv_empty[stage]" in expand
