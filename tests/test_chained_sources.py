"""The kernels launched as dependent chains (csrc/chain_launch.cuh) begin before the kernel before
them has ended. What they read is therefore not read-only for their whole life, and each has to
wait before it touches global memory. Shown on the sources: every chained kernel waits, and neither
it nor a device function it reaches reads through `const T *__restrict__` or __ldg."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_14160_gb300", "csrc")


def _closed(s, i, left, right):
    """Index after the bracket that closes the one before i."""
    depth = 1
    while depth:
        depth += (s[i] == left) - (s[i] == right)
        i += 1
    return i


def _functions():
    """name -> [(file, signature, body)] of the definitions in the CUDA sources, and the sources."""
    defs, texts = {}, {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        s = re.sub(r"//[^\n]*", "", open(path).read())
        texts[os.path.basename(path)] = s
        for m in re.finditer(r"(?<![\w.:>])(\w+)\(", s):
            end = _closed(s, m.end(), "(", ")")
            brace = re.match(r"(\s|const)*\{", s[end:])
            if brace and m.group(1) not in ("if", "for", "while", "switch", "__launch_bounds__"):
                stop = _closed(s, end + brace.end(), "{", "}")
                defs.setdefault(m.group(1), []).append((os.path.basename(path), s[m.start():end], s[end:stop]))
    return defs, texts


def _chained(defs, texts):
    """Names of the kernels launched through launch_chained or with the attribute itself."""
    names = set()
    for text in texts.values():
        for m in re.finditer(r"launch_chained\((k_\w+)", text):
            names.add(m.group(1))
    for found in defs.values():
        for _, _, body in found:
            if "launch_chained(kern" in body:   # the forms that the function chooses from
                names.update(k for k in re.findall(r"\bk_\w+", body) if k in defs)
    names.update(k for k, found in defs.items()
                 if k.startswith("k_") and any("after_previous()" in body for _, _, body in found))
    return names


def _reach(defs, start):
    seen, todo = set(), [start]
    while todo:
        n = todo.pop()
        if n in seen or n not in defs:
            continue
        seen.add(n)
        for _, _, body in defs[n]:
            todo += re.findall(r"\b(\w+)(?:<[^<>;(){}]*>)?\(", body)
    return seen


def test_chained_kernels_wait_and_read_by_plain_loads():
    defs, texts = _functions()
    names = _chained(defs, texts)
    assert {"k_factor", "k_sample", "k_eval_polar", "k_eval_broad", "k_eval", "k_eval_hulls", "k_eval_finalize",
            "k_radix_pass", "k_moments_partial", "k_cma_paths", "k_sample_reduce"} <= names
    wrong = []
    for k in sorted(names):
        reach = _reach(defs, k)
        if "after_previous" not in reach:
            wrong.append("%s does not wait" % k)
        for f in sorted(reach):
            for path, sig, body in defs[f]:
                if re.search(r"const[^,()]*\*\s*__restrict__", sig):
                    wrong.append("%s: %s, reached from %s, has a const restrict parameter" % (path, f, k))
                if "__ldg(" in body:
                    wrong.append("%s: %s, reached from %s, uses __ldg" % (path, f, k))
    assert not wrong, "\n".join(wrong)
