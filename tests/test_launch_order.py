"""Every kernel is launched while its predecessor in the stream may still run, so each has to wait for it by itself: all threads,
before any of them waits for another.  What a grid reads is promised to be visible only after its own wait; and a role that went
ahead would wait for the others on barriers, whose waits are bounded, for as long as the predecessor takes.  One kernel may
begin before its predecessor has ended, if that one lets it, having waited itself."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_00029_b200", "csrc")


def _functions(text):
    """Name, body (without its comments) of every function that starts a line and ends with a brace in the first column."""
    for m in re.finditer(r"^(?:template[^\n]*\n)?(?:__device__|__global__)[^{;]*\{\n.*?^\}", text, re.M | re.S):
        head, body = re.sub(r"//[^\n]*", "", m.group(0)).split("{\n", 1)
        yield re.findall(r"(\w+)\s*\(", re.sub(r"__launch_bounds__\([^)]*\)|__cluster_dims__\([^)]*\)", "", head))[0], body


def _own_level(body):
    """The statements of a function that stand in no block."""
    depth, kept = 0, []
    for line in body.split("\n"):
        if depth == 0:
            kept.append(line)
        depth += line.count("{") - line.count("}")
    return "\n" + "\n".join(kept)


def test_every_kernel_waits_for_its_predecessor_before_its_roles():
    kernels = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, name)) as f:
            functions = list(_functions(f.read()))
        roles = {fn: body for fn, body in functions if "mbar_wait(" in body and "__syncthreads();" not in body}
        in_roles = [fn for fn, body in roles.items() if "griddep_wait();" in body]
        # either each role of the file waits once it has its first item, which it does not have to wait for, ...
        for fn in in_roles:
            assert sorted(in_roles) == sorted(roles), (name, set(roles) - set(in_roles))
            loop = re.split(r"\n    for \((?:int w = 0)?; ?\w*;[^\n]*\{\n", roles[fn])[-1]
            assert not re.search(r"mbar_wait\(", re.split(r"        if \(w == 0\) (?:\{\s*)?griddep_wait\(\);\n", loop)[0]), (name, fn)
            assert loop.count("griddep_wait();") == 1, (name, fn)
        # ... or the kernel does, before it comes to its roles
        for fn, body in functions:
            if fn in roles or "griddep_launch_dependents();" not in body:
                assert fn in in_roles or "griddep_wait" not in body, (name, fn)
                continue
            kernels += 1
            if fn == "attn_dkdv64_kernel":  # what reads are the producer and, for the row terms, the edge warps
                assert "\n    if (threadIdx.x == 0 || (!kTerms && warp >= 12)) griddep_taken_over();\n" in _own_level(body)
                assert len(_own_level(body).split("\n    griddep_wait();")) == 2, fn
                continue
            if in_roles and any(f"{role}<" in body or f"{role}(" in body for role in in_roles):
                assert "publish_first" in body and "griddep_wait" not in body, (name, fn)
                continue
            assert len(_own_level(body).split("\n    griddep_wait();")) == 2, (name, fn)
            ahead = ("\n" + body).split("\n    griddep_wait();")[0]
            assert not re.search(r"\b(?:%s)\s*[(<]" % "|".join(["mbar_wait", *roles]), ahead), (name, fn)
        if name == "attn_dq64.cu":  # the kernel before that one lets it start when it has waited itself
            issuer = dict(functions)["dq64_mma_dq"]
            assert "            griddep_wait();\n            if (el) griddep_launch_dependents();" in issuer
            assert "    if (kDelta) griddep_launch_dependents();" in dict(functions)["dq64_body"]
        assert name == "attn_dkdv64.cu" or not any("griddep_taken_over" in body for _, body in functions), name
    assert kernels == 16, kernels
