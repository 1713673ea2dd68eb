"""Kernels that may be resident while their predecessor writes (launch_overlapped in csrc/common.cuh) read through coherent
loads only: the sources are looked at, nothing is run."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_06354_b200", "csrc")


def sources():
    return {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read()) for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def functions(text):
    """(name, head, body) of every device function and kernel."""
    for m in re.finditer(r"__(?:global|device)__[^;{}]*?(\w+)\s*\([^;{}]*\)\s*(?:const\s*)?(?=[:{])[^{;]*\{", text):
        depth, j = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        head = m.group(0)
        name = (re.findall(r"(\w+_kernel)\s*\(", head) or re.findall(r"(\w+)\s*\(", head))[0]
        yield name, head, text[m.end():j]


NON_COHERENT = re.compile(r"__ldg\s*\(|\.nc\b|\.nc\.")
CONST_RESTRICT = re.compile(r"const\s+[\w:]+\s*\*\s*__restrict__|[\w:]+\s+const\s*\*\s*__restrict__")


def test_kernels_of_overlapped_launches_wait_first_and_read_coherently():
    src = sources()
    launched = set()
    for text in src.values():
        launched |= set(re.findall(r"launch_overlapped\(\s*(?:\w+\s*==\s*\w+\s*\?\s*)?(\w+_kernel)", text)) | set(re.findall(r"launch\((\w+_kernel)", text))
    found, by_name = set(), {}
    for f, text in src.items():
        for name, head, body in functions(text):
            by_name.setdefault(name, []).append((f, head, body))
    for name, places in by_name.items():
        for f, head, body in places:
            if not name.endswith("_kernel"):
                continue
            if "pdl_wait" not in body:
                assert name not in launched, f"{f}: {name} is launched early and does not wait"
                continue
            found.add(name)
            # the kernel, and the device functions that it calls by name, to any depth
            todo, seen = [(name, f, head, body)], set()
            while todo:
                n, where, h, b = todo.pop()
                if n in seen:
                    continue
                seen.add(n)
                assert not NON_COHERENT.search(b), f"{where}: {n} (from {name}) has a non-coherent load"
                assert not CONST_RESTRICT.search(h), f"{where}: {n} (from {name}) promises that an input is read-only"
                for callee in set(re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\s*\(", b)) & set(by_name):
                    todo += [(callee, w, hh, bb) for w, hh, bb in by_name[callee] if not callee.endswith("_kernel")]
    assert launched <= found and len(found) > 25, launched - found
