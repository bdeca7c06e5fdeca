"""Grid barriers of the cooperative launches: every word that the kernels use through a
barrier pointer lies inside the words that the host allocates and clears for it."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2404_08952_gb300", "csrc")


def _read(name):
    return open(os.path.join(CSRC, name)).read()


def _value(x):
    if x.isdigit():
        return int(x)
    m = re.search(r"\b%s = (\d+)" % x, _read("common.cuh"))
    assert m, x
    return int(m.group(1))


def _words(name):
    src = _read(name)
    return [_value(x) for x in re.findall(r"\bbar \+ (\w+)", src) + re.findall(r"\bbar\[(\w+)\]", src)]


def test_words_of_the_small_mesh_steps_are_allocated():
    m = re.search(r"upload\(m, std::vector<unsigned>\((\w+), 0u\), &bar\)", _read("api.cu"))
    words = _words("kernels.cuh")
    assert len(words) >= 5
    assert max(words) < _value(m.group(1))


def test_words_of_the_batch_lie_in_the_cleared_head_of_the_workspace():
    off = int(re.search(r"b\.bar = reinterpret_cast<unsigned \*>\(B\(ws, L\.status \+ (\d+)\)\)", _read("api.cu")).group(1))
    assert off + 4 * (max(_words("kernels.cuh")) + 1) <= 1024


def test_a_block_takes_one_answer_from_the_abort_word():
    """What a block does after reading the abort word leads to block barriers, so one thread
    reads it for the block (grid_aborted, or thread 0 of a barrier); only a poll whose
    answer goes through shared memory reads it by itself."""
    for name in ("kernels.cuh", "implicit.cu"):
        src = _read(name)
        reads = [src[:m.start()].rsplit("\n", 1)[1] for m in re.finditer(r"\*\(volatile unsigned \*\)\([^()]*\)(?! =)", src)]
        assert all(r.strip() == "if ((it & 63u) == 0 &&" for r in reads), (name, reads)
        assert "grid_aborted(" in src


def test_words_of_the_solver_lie_in_its_control_block():
    src = _read("api.cu")
    ctrl = int(re.search(r"kImpCtrl = (\d+)", src).group(1))
    first = int(re.search(r"imp->bar = reinterpret_cast<unsigned \*>\(reinterpret_cast<char \*>\(imp->scal\) \+ (\d+)\)",
                          src).group(1))
    status = int(re.search(r"a\.status = imp->bar \+ (\d+)", src).group(1))
    words = _words("implicit.cu")
    assert first + 4 * (max(words + [status]) + 1) <= ctrl
    assert status not in words
