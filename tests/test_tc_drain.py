"""A tensor-core kernel's CTA does not end under its own asynchronous copies and
MMAs, also when one of its bounded waits gave up: the thread that issues them
waits for them after its loop, on every path."""
import glob
import os
import re

from paper_2211_14318_gb300 import build as b


def _kernels():
    """(name, body) of every kernel that issues copies or MMAs."""
    for path in sorted(glob.glob(os.path.join(b.CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", src):
            i = src.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
            body = src[i:j]
            if re.search(r"\b(tma_load_2d|bulk_load|umma_bf16)\(", body):
                yield m.group(1), body


def _unconditional(body: str, call: str) -> bool:
    """The call stands in the issuing lane's block itself, not in a branch on
    whether a wait gave up."""
    stack, start = [], 0
    for m in re.finditer(r"[{};]|\b%s\(" % call, body):
        t = m.group()
        if t == "{":
            stack.append(body[start:m.start()])
        elif t == "}":
            stack.pop()
        if t in "{};":
            start = m.end()
        elif "lane == 0" in stack[-1] or "threadIdx.x == 0" in stack[-1]:
            return body[start:m.start()].strip() == ""
    return False


def test_issuing_threads_wait_for_their_copies_and_mmas():
    names = set()
    for name, body in _kernels():
        names.add(name)
        assert _unconditional(body, "drain_copies"), f"{name}: copies"
        assert _unconditional(body, "drain_mmas"), f"{name}: MMAs"
    assert names == {"k_gemm", "k_gemm_ws", "k_mlp_forward", "k_mlp_train", "k_mlp_dw"}
