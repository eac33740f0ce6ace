"""CPU: rules of the CUDA sources that no launch on a healthy single GPU shows,
read from the text of the sources."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_28637_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_noalloc_checks_its_launches_before_psi_is_multiplied():
    """A chain that failed leaves an earlier call's factor in the scratch."""
    run = source("roks_noalloc.cu")
    run = run[run.index("cholesky_inverse(nb"):run.index("k_rows_times_upper<T><<<")]
    assert re.search(r"if \(cudaGetLastError\(\) != cudaSuccess\) return broken\(flag, st\);", run)
    # and no way out between them leaves the status flag set for the next call
    assert "return ROKS_ECUDA" not in run


def test_the_potentials_bound_is_cleared_only_where_they_are_written():
    """An energies-only call keeps the potentials, and must keep their bound,
    from which the apply takes its scale: the plane pass clears it."""
    grid = source("k_grid.cu")
    body = grid[grid.index("void potentials(int N"):]
    body = body[:body.index("\n}\n")]
    assert re.search(r"a\.vmax = energies_only \? nullptr : vmax;", body)
    assert len(re.findall(r"\bvmax\b", body)) == 3       # the parameter and that line


def test_shared_memory_is_asked_for_in_every_context():
    """The limit belongs to the context of the current device: a flag that
    remembers having asked refuses the launches on the next device."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = source(os.path.basename(path))
        calls = len(re.findall(r"cudaFuncSetAttribute\(", text))
        assert calls == (1 if path.endswith("k_stream.cu") else 0), path
        # no flag stands before the asking
        assert not re.search(r"static bool \w+ = false;", text), path


def test_copies_in_assembly_are_ordered_with_memory():
    """Without the clobber the compiler may move the reads of a ring's slot past
    the copy that overwrites it."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = source(os.path.basename(path))
        for m in re.finditer(r"asm volatile\(", text):
            depth, i = 1, m.end()
            while depth:                                   # to the closing parenthesis
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            body = text[m.end():i]
            if "cp.async" in body:
                assert '"memory"' in body, (path, body)
