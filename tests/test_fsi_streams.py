"""The streams of a coupled step (ibfsa_fsi_step), on the CPU: the plate's host code is linked with a
CUDA runtime that only logs (fake_cudart.cpp).  Work on another stream than the caller's has to wait for
what it reads, and the caller's stream has to wait for it: before the next step, and before the call
returns, whatever call fails on the way (an unjoined stream leaves work that nothing orders with the
caller's next use of the memory, and ends a capture in an error).  The other stream has the priority of the
caller's, and where that belongs to a green context, whose part of the chip a stream of the runtime does
not keep to, everything stays on the caller's.
"""
import os
import subprocess

import pytest

from paper_1905_00182_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    try:
        cc = B.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    out = str(tmp_path_factory.mktemp("fsi") / "fsi_streams")
    r = subprocess.run([cc, *B.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "--cudart",
                        "none", "-I", B.CSRC, "-I", os.path.join(os.path.dirname(B.HERE), "include"),
                        os.path.join(HERE, "fake_cudart.cpp"), os.path.join(B.CSRC, "plate.cu"),
                        "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def _run(program, fail=-1, steps=2, priority=0, green=0):
    r = subprocess.run([program, str(fail), str(steps), str(priority), str(green)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lines = [x.split() for x in r.stdout.splitlines()]
    assert lines[-1][0] == "returned"
    created = [int(x[2]) for x in lines if x[0] == "stream"]  # priorities
    return [x for x in lines if x[0] != "stream"][:-1], int(lines[-1][1]), created


def _reaches(log, i, stream):
    """positions from which on `stream` is ordered behind entry i of the log (None: never)"""
    record = log[i][0] == "record"
    at = {log[i][2 if record else 1]: i}   # stream -> from where it is ordered behind entry i
    events = {log[i][1]} if record else set()
    for k in range(i + 1, len(log)):
        if log[k][-1] == "FAILED":
            continue
        op, a = log[k][0], log[k][1]
        if op == "record":
            events.discard(a)
            if log[k][2] in at:
                events.add(a)
        elif op == "wait" and log[k][2] in events:
            at.setdefault(a, k)
        elif op == "sync" and a in at:
            at.setdefault(stream, k)
    return at.get(stream)


def test_order_of_a_coupled_step(program):
    log, rc, _ = _run(program)
    assert rc == 0
    work = [k for k, x in enumerate(log) if x[0] == "launch"]
    per = len(work) // 2
    assert per == 8  # markers, three stages, three force averages, the plate's step
    names = ["markers", "stage 1", "average 1", "stage 2", "average 2", "stage 3", "average 3", "plate"]
    at = {(s, n): work[s * per + j] for s in range(2) for j, n in enumerate(names)}

    def before(a, b):
        k = _reaches(log, a, log[b][1])
        return k is not None and k < b or log[a][1] == log[b][1] and a < b

    for s in range(2):
        for j, n in enumerate(names[:-1]):
            if n == "stage 3":  # the plate waits for its forces (the event), not for its end
                rec, average = at[s, n] + 1, at[s, "average 3"]
                assert log[rec][0] == "record" and _reaches(log, rec, log[average][1]) < average
            else:
                assert before(at[s, n], at[s, names[j + 1]]), (s, n)
    for n in names:
        assert before(at[0, n], at[1, "markers"]), n


def test_every_failure_leaves_the_streams_joined(program):
    n = len(_run(program)[0])
    for fail in range(n):
        log, rc, _ = _run(program, fail)
        assert rc < 0
        assert sum(x[-1] == "FAILED" for x in log) == 1
        for k, x in enumerate(log):
            if x[0] == "launch" and x[-1] != "FAILED" and x[1] != "main":
                assert _reaches(log, k, "main") is not None, (fail, k, log)


@pytest.mark.parametrize("priority", [0, -2, -5])
def test_side_stream_has_the_priority_given(program, priority):
    _, rc, created = _run(program, priority=priority)
    assert rc == 0 and created == [priority]


def test_in_line_in_a_green_context(program):
    log, rc, created = _run(program, green=1)
    assert rc == 0 and created == []
    assert len(log) == 16 and all(x[:2] == ["launch", "main"] for x in log)
