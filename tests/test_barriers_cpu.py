"""Every __syncthreads() of the device code stands where all threads of a CTA come by:
not in a branch on a thread's place or role (CUDA defines the barrier only for
conditions that are uniform over the CTA, also where both arms hold one).  Conditions
on the place are told by the names the sources use for it."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PLACE = re.compile(r"\b(threadIdx|tid|lane|warp|owner|halo)\b")


def _divergent_barriers(text):
    text = re.sub(r"//[^\n]*|/\*.*?\*/", lambda m: " " * len(m.group()), text, flags=re.S)
    out, stack, last_if = [], [], {}
    start = 0  # of the statement or block header being read
    depth = 0  # of parentheses: the semicolons of a for header end no statement
    for m in re.finditer(r"[{}();]|__syncthreads", text):
        t = m.group()
        if t == "(" or t == ")":
            depth += 1 if t == "(" else -1
        elif t == "{":
            head, level = text[start:m.start()].strip(), len(stack)
            cond = head
            if re.search(r"\belse$", head):
                cond = last_if.get(level, "")
            elif re.search(r"\bif\b", head):
                last_if[level] = head
            elif not re.search(r"\b(for|while)\b", head):
                cond = ""
            stack.append(bool(re.search(r"\b(if|else|for|while)\b", head) and PLACE.search(cond)))
            start = m.end()
        elif t == "}":
            stack.pop()
            start = m.end()
        elif t == ";":
            if depth == 0:
                start = m.end()
        else:
            head = text[start:m.start()]
            if any(stack) or (re.search(r"\b(if|else)\b", head) and PLACE.search(head)):
                out.append(text.count("\n", 0, m.start()) + 1)
    return out


def test_no_barrier_in_a_role():
    files = glob.glob(os.path.join(ROOT, "paper_2303_03026_gb300", "csrc", "*.cu*"))
    assert len(files) > 10
    bad = {os.path.basename(f): _divergent_barriers(open(f).read()) for f in files}
    assert not {f: lines for f, lines in bad.items() if lines}


def test_the_reader_finds_them():
    ok = "for (int i = threadIdx.x; i < n; i++) { x(); }\n__syncthreads();\nif (n) { __syncthreads(); }"
    assert _divergent_barriers(ok) == []
    assert _divergent_barriers("if (owner) {\n f();\n __syncthreads();\n} else {\n __syncthreads();\n}") == [3, 5]
    assert _divergent_barriers("if (tid < 4) __syncthreads();") == [1]
    assert _divergent_barriers("for (int i = tid; i < n; i += 32) {\n if (n) {\n __syncthreads(); } }") == [3]
