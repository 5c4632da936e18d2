"""Every launch that sets the dependent-launch attribute, whatever it names its
kernel by: the kernel waits (griddepcontrol.wait) before it touches memory.

A kernel launched so may run beside the kernel before it, and only its wait
orders the two.  The launches are found in the sources: each call of
launch_config whose last argument is true, and each function that writes the
attribute itself.  The kernel is resolved from `kernel()` of the launcher, from
`&name`, or from the local variable that holds it; a launch that cannot be
resolved fails.  Before the wait a kernel may ask for data to be brought into
L2 (prefetch_l2) and look at an address, nothing else."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1502_02389_gb300", "csrc")
REQUIRED = {"reduce_ldg", "reduce_tma", "combine_kernel", "combine64_kernel", "comp_reduce",
            "mixed_reduce", "unaligned_reduce", "unaligned_map", "scal_ldg", "scal_tma", "axpy_ldg",
            "bs_map", "gemv_warp", "gemv_warp_rows", "gemv_split_rows", "gemv_tma", "gemv_t_kernel",
            "gemv_t_staged", "gemv_t_cols", "gemv_t_combine", "gemv_t_combine_cols",
            "mlp_forward_fused", "masked_mse", "mlp_back_rows", "mlp_weight_grads", "adam"}


def sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as fh:
                yield f, re.sub(r"//[^\n]*", "", fh.read())


def closing(text, i, pair):
    """Index of the bracket that closes the one at i."""
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == pair[0]) - (text[j] == pair[1])
        if depth == 0:
            return j
    raise AssertionError("unbalanced " + pair)


def arguments(text):
    out, depth, start = [], 0, 0
    for i, c in enumerate(text):
        depth += (c in "([{") - (c in ")]}")
        if c == "," and depth == 0 and text[start:i].count("<") == text[start:i].count(">"):
            out.append(text[start:i].strip())
            start = i + 1
    return out + [text[start:].strip()]


def names_in(expr):
    return set(re.findall(r"&(\w+)\s*(?=[<)])", expr))


def dependent_kernels():
    found = {}
    for f, text in sources():
        for m in re.finditer(r"\blaunch_config\(", text):
            end = closing(text, m.end() - 1, "()")
            args = arguments(text[m.end():end])
            if args[-1] != "true":
                continue
            assert len(args) == 8, (f, args)
            k, where = args[0], f"{f}: launch_config({args[0]}"
            if k == "kernel()":
                at = text.rfind("static const void* kernel()", 0, m.start())
                brace = text.index("{", at)
                names = names_in(text[brace:closing(text, brace, "{}")])
            elif re.fullmatch(r"\w+", k):
                sets = [s for s in re.finditer(r"\b" + k + r"\s*=([^;]*);", text[:m.start()])]
                assert sets, where
                names = names_in(sets[-1].group(1))
            else:
                names = names_in(k)
            assert names, where
            for n in names:
                found.setdefault(n, where)
        for m in re.finditer(r"cudaLaunchAttributeProgrammaticStreamSerialization", text):
            seg = text[text.rfind("\n}", 0, m.start()):text.find("\n}", m.start())]
            if "lift_status launch_config(" in seg:
                continue
            names = names_in(seg)
            assert names, (f, seg[-300:])
            for n in names:
                found.setdefault(n, f)
    return found


def kernels():
    """name -> [(pointer parameters, body)]"""
    out = {}
    for _, text in sources():
        for m in re.finditer(r"__global__", text):
            head = re.compile(r"\s*void\s*(?:__launch_bounds__\s*\()?").match(text, m.end())
            i = head.end()
            if "__launch_bounds__" in head.group(0):
                i = closing(text, i - 1, "()") + 1
            sig = re.compile(r"\s*(\w+)\s*\(").match(text, i)
            close = closing(text, sig.end() - 1, "()")
            brace = re.compile(r"\s*\{").match(text, close + 1)
            if not brace:                      # a declaration
                continue
            params = re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)\s*(?:,|$)", text[sig.end():close] + ",")
            body = text[brace.end():closing(text, brace.end() - 1, "{}")]
            out.setdefault(sig.group(1), []).append((params, body))
    return out


ACCESS = re.compile(r"\b(ld_\w+|st_stream|__ldg|__ldcg|bulk_g2s|bulk_s2g|cp4|cp16|cp_flat|copy16|"
                    r"atomic\w+|fold_\w+|load)\s*[<(]")


def test_every_dependent_launch_is_resolved_and_waits_first():
    found, bodies = dependent_kernels(), kernels()
    assert REQUIRED <= set(found), REQUIRED - set(found)
    for name, where in sorted(found.items()):
        assert name in bodies, (name, where)
        for params, body in bodies[name]:
            wait = body.find("pdl_wait()")
            assert wait >= 0, f"{name} ({where}) is launched as a dependent and never waits"
            head = re.sub(r"__shared__[^;]*;", "", body[:wait])
            while "prefetch_l2(" in head:
                i = head.index("prefetch_l2(")
                head = head[:i] + head[closing(head, i + len("prefetch_l2(") - 1, "()") + 1:]
            assert not ACCESS.search(head), (name, ACCESS.search(head).group(0))
            assert not re.search(r"\bjob\.(L|R|out|bias)\b", head), name
            for p in params:
                assert not re.search(r"\b" + p + r"\s*\[|(?<![\w)\]])\s\*\s*" + p + r"\b", head), (name, p)


def test_the_check_sees_a_missing_wait():
    # the check itself, on a kernel that reads first
    bad = "int i = threadIdx.x; float v = x[i]; pdl_wait(); y[i] = v;"
    head = bad[:bad.find("pdl_wait()")]
    assert re.search(r"\bx\s*\[", head)
    assert ACCESS.search("const float v = __ldg(x + i);")
