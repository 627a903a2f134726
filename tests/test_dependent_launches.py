"""Rules of the kernels launched with programmatic serialization, read from the CUDA sources: such a
kernel runs beside its predecessor until pdl_wait(), so its launch must not end before it, and nothing
the predecessor writes may be promised to the compiler as read-only or unaliased."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_21908_gb300", "csrc")


def _sources():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            out[os.path.basename(path)] = re.sub(r"//[^\n]*", "", f.read())
    return out


def _block(text, start, op="{", cl="}"):
    """text from the first `op` after start to its matching `cl`, without both."""
    i = text.index(op, start)
    depth, j = 0, i
    while True:
        depth += {op: 1, cl: -1}.get(text[j], 0)
        if depth == 0:
            return text[i + 1:j]
        j += 1


def dependent_kernels():
    """name -> (parameter list, body) of every kernel that launch_pdl launches."""
    src = _sources()
    names = set()
    for text in src.values():
        for m in re.finditer(r"launch_pdl\(\s*(\w+)", text):
            if m.group(1).startswith("k_"):
                names.add(m.group(1))
            else:  # a local function pointer, the nearest above: auto kf = [cond ?] k_name<...> [: ...];
                names.add(re.findall(r"auto %s =[^;]*?\b(k_\w+)" % m.group(1), text[:m.start()])[-1])
    assert len(names) >= 15
    out = {}
    for name in names:
        for text in src.values():
            m = re.search(r"__global__[^;{]*?\b%s\s*\(" % name, text)
            if m:
                out[name] = (_block(text, m.end() - 1, "(", ")"), _block(text, m.end()))
    assert set(out) == names
    return out


def test_no_block_leaves_before_its_predecessor():
    """Before the first unconditional pdl_wait() a block returns only behind a pdl_wait() of its own; the
    bound of a thread's index is no such return (the first thread of every block is in range)."""
    for name, (_, body) in dependent_kernels().items():
        assert "pdl_wait();" in body, name
        for m in re.finditer(r"pdl_wait\(\);|\breturn;", body):
            if m.group(0) == "return;":
                stmt = body[max(body.rfind(c, 0, m.start()) for c in ";{}") + 1:m.end()].strip()
                before = body[body.rfind("{", 0, m.start()) + 1:m.start()]
                guard = re.fullmatch(r"if \(\w+ >= \w+\) return;", stmt)
                assert guard or before.strip().endswith("pdl_wait();"), (name, stmt)
            elif not re.match(r"\s*return;", body[m.end():]):
                break


# Written when a handle is created, before any launch of the chain: twiddles, weights, projector rows and
# blocks, the local potential.  The Poisson kernels' twiddles may be written by the first of them.
CREATED = {"twg", "wf", "rows", "vloc", "Dmat"}


def test_what_a_predecessor_writes_is_not_promised_read_only():
    for name, (params, body) in dependent_kernels().items():
        allowed = set() if name.startswith("k_poisson") else CREATED
        assert set(re.findall(r"__restrict__\s+(\w+)", params)) <= allowed, name
        assert "__ldg(" not in body, name


def test_launchers_keep_no_unsynchronised_state():
    """What a launcher remembers between calls (opted-in kernels, waves of a device) is shared by host
    threads and devices: per-device atomics, no plain variable."""
    for file, text in _sources().items():
        local = re.findall(r"^[ \t]+static\s+(?!const\b|constexpr\b|std::atomic\b)[^;({]*[;={]", text, re.M)
        assert not local, (file, local)
