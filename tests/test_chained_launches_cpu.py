"""Every kernel launched with the programmatic-serialization attribute waits for the kernel
before it, ahead of anything else it does.  A missing wait is a race that a run cannot be
relied on to show, so the sources are read: the kernels named in launch_chained() calls
(directly, or through the variable that selects a variant), and the first statement of each."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2301_09710_gb300" / "csrc"


def _text(path):
    t = re.sub(r"/\*.*?\*/", " ", path.read_text(), flags=re.S)
    t = re.sub(r"//[^\n]*", " ", t)
    return t.replace("\\\n", " \n")


SOURCES = {p.name: _text(p) for p in sorted(CSRC.glob("*.cu")) + sorted(CSRC.glob("*.cuh"))}


def _first_argument(text, at):
    """The first argument of the call whose opening parenthesis is at `at`."""
    depth = 0
    for n in range(at, len(text)):
        c = text[n]
        depth += c in "(<" and 1 or 0
        depth -= c in ")>" and 1 or 0
        if (c == "," and depth == 1) or depth == 0:
            return text[at + 1:n].strip()
    raise AssertionError("unbalanced call")


def chained_kernels():
    names = {}
    for src, text in SOURCES.items():
        for m in re.finditer(r"\blaunch_chained\s*\(", text):
            if re.match(r"launch_chained\s*\(\s*void\s*\(", text[m.start():]):
                continue  # its definition
            arg = _first_argument(text, m.end() - 1)
            found = re.findall(r"\bk_\w+", arg)
            if not found:  # a variable: the kernels its nearest initialiser chooses from
                init = [i for i in re.finditer(r"\bauto\s+%s\s*=([^;]*);" % re.escape(arg), text) if i.start() < m.start()]
                assert init, f"{src}: launch_chained({arg}, ...): cannot tell which kernel"
                found = re.findall(r"\bk_\w+", init[-1].group(1))
            assert found, f"{src}: launch_chained({arg}, ...) names no kernel"
            for k in found:
                names.setdefault(k, src)
    return names


def body(kernel):
    """The text of the kernel's body, from behind its opening brace."""
    found = []
    for text in SOURCES.values():
        for m in re.finditer(r"\b%s\s*\(" % kernel, text):
            head = text[max(0, m.start() - 300):m.start()]
            if "__global__" not in head or re.search(r"[;}]", head[head.rindex("__global__"):]):
                continue
            depth, n = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[n], 0)
                n += 1
            rest = text[n:].lstrip()
            if rest.startswith("{"):
                found.append(rest[1:])
    assert len(found) == 1, f"{kernel}: {len(found)} definitions"
    return found[0]


def test_every_chained_kernel_waits_first():
    kernels = chained_kernels()
    # the kernels of a step, so that a call this test cannot read does not pass unseen
    assert {"k_transpose", "k_mubar_cache", "k_rot_fwd", "k_rot_patch", "k_fwd_sep_fused", "k_fwd_dir_fused", "k_fwd_reduce",
            "k_pad_rows", "k_adj_sep_fused", "k_adj_dir_fused", "k_adj_gather", "k_adj_rot_t"} <= set(kernels)
    late = []
    for k in sorted(kernels):
        stmts = [s.strip() for s in body(k).split(";")]
        # names, constants and shared arrays touch no global memory
        while re.match(r"(using|constexpr|(extern\s+)?__shared__)\b", stmts[0]):
            stmts.pop(0)
        if stmts[0] != "wait_previous_kernel()":
            late.append(k)
    assert not late, f"no wait for the previous kernel ahead of everything else: {late}"


def test_the_attribute_is_set_in_one_place():
    hits = [src for src, t in SOURCES.items() for _ in re.finditer("ProgrammaticStreamSerialization\\b", t)]
    assert hits == ["spect_internal.cuh"], hits
    # and no kernel lets its successor start before its own writes are done
    assert not any("launch_dependents" in t or "cudaTriggerProgrammaticLaunchCompletion" in t for t in SOURCES.values())
