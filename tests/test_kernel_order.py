"""Orders inside kernels that no run can show to be missing: read from the
sources, since a late access would have to be provoked on a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_03640_gb300", "csrc")


def _body(name, kernel):
    """The text of a kernel, without comments."""
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    at = text.index("{", re.search(r"\b%s\s*\(" % kernel, text).end())
    depth = 0
    for end in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        if depth == 0:
            return text[at:end]


def test_step_scalars_are_read_before_the_block_is_counted():
    """k_solo_steps: the block that counts last writes steps_done, so every
    thread's read of it has to be ordered before its own block's count, that
    is, to lie before the last barrier ahead of it (thread 0's own apart)."""
    body = _body("k_solo.cu", "k_solo_steps")
    count = body.index("atomicAdd(&sc->counter")
    barrier = body.rindex("__syncthreads()", 0, count)
    assert "steps_done" not in body[barrier:count]
    assert "sc->p1" not in body[barrier:count] and "sc->p2" not in body[barrier:count]
    # and the scalars are written behind the barrier that follows the count
    write = body.index("sc->steps_done =")
    assert "__syncthreads()" in body[count:write]


def test_dense_batch_is_read_behind_the_wait():
    """k_dense_convert may start while the kernel that writes its batch still
    runs: it waits, and then reads the batch by ordered loads only, never
    through the read-only cache."""
    body = _body("k_dense.cu", "k_dense_convert")
    wait = body.index("grid_dep_wait()")
    assert "cost[" not in body[:wait] and "pack_transpose" not in body[:wait]
    pack = _body("k_dense.cu", "pack_transpose")
    assert pack.count("src") == 1 and "ld_ordered(src" in pack


def test_gradient_scale_is_read_behind_the_wait():
    """The caller's kernel that writes the scale of msat_backward is the one
    before the variable pass in the stream: every read of it is an ordered
    load, which stays behind the pass's wait."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "k_step.cu")).read())
    assert not re.search(r"gscale\s*\[|\*\s*gscale\b(?!,|\))", text)
    assert "ld_ordered(gscale + " in text


def test_parts_of_a_batch_are_counted_in_64_bits():
    """launch_eval_sparse takes a batch in parts: the position behind the last
    part of a batch of nearly 2^31 assignments is past 32 bits."""
    body = _body("k_eval.cu", "cudaError_t launch_eval_sparse")
    loops = re.findall(r"for \((.*?) b0 = 0;", body)
    assert loops == ["long long", "long long"]
