"""What the kernels' sources leave out, because no run can show that it is absent."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_02868_gb300", "csrc")


def _code(path):
    """The source without its comments."""
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


def test_shuffles_name_their_lanes():
    # __activemask() is whatever lanes happen to run together: after a loop or branch that
    # differs by lane, a shuffle over it may leave out lanes that it should read
    files = glob.glob(os.path.join(CSRC, "*.cu*"))
    assert files and not [os.path.basename(f) for f in files if "__activemask" in _code(f)]


def _function(code, name):
    """Body of the function `name` defined in code."""
    start = re.search(r"\b%s\([^;{]*\)\s*\{" % name, code).end()
    depth, i = 1, start
    while depth:
        depth += {"{": 1, "}": -1}.get(code[i], 0)
        i += 1
    return code[start:i]


def test_every_exit_leaves_the_exchange_buffers_marked():
    # A call may leave its coarse solves anywhere (an error, a wait that gave up on the other
    # right-hand side of a pair): the tagged exchange words are good only after an end_coarse
    # that saw no timeout, so nothing but begin_coarse clears them and nothing but these two
    # decides whether they are good, and a call ends the coarse solves of all its handles
    # before it reports a timeout.
    code = "".join(_code(f) for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    begin, end = _function(code, "mg_status begin_coarse"), _function(code, "mg_status end_coarse")
    assert "cdirty = true" in begin and "cdirty = cs->timeouts != 0" in end
    rest = code.replace(begin, "").replace(end, "")
    assert "cdirty" not in rest and not re.search(r"Memset\w*\([^;]*(cepoch|crows|cpart|cstats)", rest)
    for name in ("mg_status solve_rhs_pairs", "mg_status solve_rhs", "mg_status mg_coarse_solve"):
        body = _function(code, name)
        assert "begin_coarse(" in body and "MG_ETIMEOUT" not in body[body.index("begin_coarse("):body.index("end_coarse(")]
        loop = re.search(r"for \([^;]*Hp : \{&A, &Bh\}\) \{", body)
        if loop:
            depth, i = 1, loop.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(body[i], 0)
                i += 1
            assert "end_coarse(" in body[loop.end():i] and "return" not in body[loop.end():i]
