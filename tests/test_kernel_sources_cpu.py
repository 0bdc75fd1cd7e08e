"""Rules of the kernel sources that no output shows until a compiler makes use of them: read from the sources themselves."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_01460_b200", "csrc")


def _sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
        yield os.path.basename(path), re.sub(r"//[^\n]*", "", text)


def _closing(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced")


def _kernels():
    """(file, name, parameter list, body) of every __global__ function that is defined in the sources."""
    for name, text in _sources():
        for m in re.finditer(r"__global__\b", text):
            at = m.end()
            while True:  # return type and attributes, then the name in front of the parameter list
                word = re.compile(r"\s*(\w+)\s*").match(text, at)
                at = word.end()
                if word.group(1).startswith("__"):
                    at = _closing(text, at, "()") + 1
                elif word.group(1) != "void":
                    break
            close = _closing(text, at, "()")
            start = text.index("{", close)
            yield name, word.group(1), text[at:close], text[start:_closing(text, start, "{}") + 1]


def test_every_kernel_is_found():
    names = [k for _, k, _, _ in _kernels()]
    assert len(names) == len(set(names)) == sum(t.count("__global__") for _, t in _sources())
    assert {"rollout_tc_kernel", "gae_kernel_v4", "critic_kernel", "ppo_net_tc_kernel", "adam_kernel"} <= set(names)


@pytest.mark.parametrize("file,name,params,body", [pytest.param(*k, id=k[1]) for k in _kernels() if "wait_for_predecessor()" in k[3]])
def test_a_dependent_kernel_declares_nothing_constant_that_its_predecessor_may_write(file, name, params, body):
    assert "__restrict__" not in params, f"{file}: {name}"
    assert not re.search(r"\b__ldg\s*\(", body), f"{file}: {name}"


def test_no_load_takes_the_non_coherent_path_by_hand():
    for name, text in _sources():
        assert "ld.global.nc" not in text, name


def test_inline_assembly_that_reads_memory_is_kept_in_order():
    """Without `volatile` an asm statement is a pure function of its operands: a load may then move over the wait for what it
    reads, or be done once for several uses."""
    for name, text in _sources():
        for m in re.finditer(r"\basm\s*\(", text):  # (asm volatile does not match)
            statement = text[m.start():_closing(text, m.end() - 1, "()")]
            assert not re.search(r"\b(ld|tcgen05\.ld|ldmatrix|atom|red|st|mbarrier)\b", statement), (name, statement[:120])


def test_the_update_kernel_lets_its_weight_image_land_when_it_gives_up():
    """The image comes on two barriers.  A role that gives up may have waited for neither; the block must, before it leaves."""
    body = {k: b for _, k, _, b in _kernels()}["ppo_net_tc_kernel"]
    end = body[body.index("__syncthreads_and(ok)"):]
    assert re.search(r"mbar_wait\(bar_load, 0\)", end) and re.search(r"mbar_wait\(bar_load \+ 8, 0\)", end)


def test_head_derivatives_have_been_read_before_their_next_writer_is_let_on():
    """The update kernel of H <= 128 keeps one tile of head derivatives for two tiles of rows in flight.  The loss that writes it waits
    for the logits' products only, and a commit covers what was issued before it: no product that reads the tile may be issued
    between that commit and the end of a turn."""
    body = {k: b for _, k, _, b in _kernels()}["ppo_net_tc_kernel"]
    reads = [m.start() for m in re.finditer(r"AT16\(dhead\)", body)]
    writer = body.index("product(kLogits, s)")
    commit = body.index("mma_commit(done0 + 8 * kLogits)")
    assert len(reads) >= 2 and commit < writer
    assert all(at < commit for at in reads), "a product that reads the tile is behind the commit its writer waits for"
