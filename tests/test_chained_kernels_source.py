"""A kernel started by launch_next may be resident while the kernel before it
still writes.  Read as text: such kernels wait before anything else, and
neither they nor the device functions they share read through the read-only
path (``.nc``, ``__ldg``, or ``__restrict__`` pointers, which allow the compiler
to choose it)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_01294_gb300", "csrc")
# files whose kernels are launched the ordinary way only, and the read-only loads kept for them
ORDINARY = ("gz_adjoint.cu", "gz_api.cu", "gz_noalloc.cu", "gz_peaks.cu")
READ_ONLY = ("load_row32", "load4")


def _sources():
    return {os.path.basename(f): open(f).read() for f in glob.glob(os.path.join(CSRC, "*.cu*"))}


def _match(s, a, pair):
    """End of the bracketed text that opens at a."""
    depth, k = 0, a
    while True:
        depth += (s[k] == pair[0]) - (s[k] == pair[1])
        k += 1
        if depth == 0:
            return k


def _functions(s, kind):
    """(name, parameters, body) of every function with the given qualifier."""
    for m in re.finditer(kind + r"\b", s):
        b = m.end()
        while True:
            f = re.compile(r"(\w+)\s*\(").search(s, b)
            a, b = f.end() - 1, _match(s, f.end() - 1, "()")
            if f.group(1) not in ("__launch_bounds__", "__align__"):
                break
        rest = s[b:].lstrip()
        if ";" in s[m.end():a] or not rest.startswith(("{", "const {")):
            continue  # (a declaration, or an array)
        c = s.index("{", b)
        yield f.group(1), s[a:b], s[c:_match(s, c, "{}")]


def test_chained_kernels_wait_first_and_take_no_restricted_pointers():
    chained = set()
    for name, s in _sources().items():
        if name in ORDINARY:
            assert "launch_next" not in s, name
            continue
        for fn, sig, body in _functions(s, "__global__"):
            if body[1:].lstrip().startswith("after_previous();"):
                chained.add(fn)
                assert "__restrict__" not in sig, (name, fn)
            else:
                assert not re.search(r"\b(launch_next\(c, |one\(|go\(|group\()" + fn + r"\b", s), (name, fn)
    assert len(chained) > 40  # (the parser finds them)


def test_shared_device_functions_keep_off_the_read_only_path():
    for name, s in _sources().items():
        for fn, sig, body in _functions(s, "__device__"):
            bad = any(w in body for w in (".nc.", "__ldg"))
            if name in ORDINARY:
                continue
            if fn in READ_ONLY:
                users = {f for f, t in _sources().items() if re.search(r"\b" + fn + r"\b\s*[<(]", t)}
                assert users <= {name, "gz_adjoint.cu"}, (fn, users)
                continue
            assert not bad and "__restrict__" not in sig and "__restrict__" not in body, (name, fn)
            for m in re.finditer(r'asm\s*(volatile)?\s*\("ld\.', body):
                assert m.group(1), (name, fn)
