"""Source check (no GPU): kernels that may start before the kernel ahead of them
has finished (they call dependency_wait()) read what other kernels write through
plain loads.

The read-only path (__ldg, or const __restrict__ parameters, which let the
compiler take it) asks that the data does not change while the kernel runs. A
kernel that starts early breaks that for everything its predecessors write, and
no test of results can be relied on to notice, so the sources are read instead:
in such kernels and in the device functions that they call, only the kernel
matrix B, the source matrices and tables in shared memory may use it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_10070_gb300", "csrc")
READ_ONLY = {"B", "src2", "bin"}  # the kernel matrix, source matrices, a table in shared memory


def functions():
    """(kind, name, parameters, body) of every __global__ and __device__ function."""
    def close(s, i, pair):  # the position after the bracket that s[i] opens
        depth = 0
        while True:
            depth += {pair[0]: 1, pair[1]: -1}.get(s[i], 0)
            i += 1
            if depth == 0:
                return i

    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        s = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__(global|device)__", s):
            at = m.end()
            bounds = re.compile(r"[\s\w]*__launch_bounds__(?=\()").match(s, at)
            if bounds:
                at = close(s, bounds.end(), "()")
            head = re.compile(r"[\s\w<>,:&*]*?(\w+)(?=\()").match(s, at)
            if not head:
                continue  # a variable
            end = close(s, head.end(), "()")
            if not s[end:].lstrip().startswith("{"):
                continue
            start = s.index("{", end)
            out.append((m.group(1), head.group(1), s[head.end() + 1:end - 1], s[start:close(s, start, "{}")]))
    return out


def violations(params, body):
    bad = [p.split()[-1] for p in params.split(",") if "__restrict__" in p]
    roots = dict(re.findall(r"\*\s*(\w+)\s*=\s*(?:reinterpret_cast<[^>]*>\()?([\w.>-]+)", body))
    for arg in re.findall(r"__ldg\((\w+)", body):
        bad.append(arg if arg in READ_ONLY else roots.get(arg, arg))  # a row pointer counts as what it points into
    return sorted({b for b in bad if b not in READ_ONLY})


def test_dependent_kernels_read_written_data_by_plain_loads():
    fns = functions()
    kernels = [f for f in fns if f[0] == "global" and "dependency_wait()" in f[3]]
    assert len(kernels) >= 14, [k[1] for k in kernels]
    device = {f[1]: f for f in fns if f[0] == "device"}
    bad = {}
    for _, name, params, body in kernels:
        todo, seen = [(params, body)], set()
        while todo:
            p, b = todo.pop()
            for v in violations(p, b):
                bad.setdefault(name, set()).add(v)
            for callee in set(re.findall(r"\b(\w+)(?:<[\w ]+>)?\(", b)) & set(device) - seen:
                seen.add(callee)
                todo.append(device[callee][2:])
    assert not bad, bad


def test_every_kernel_launched_early_waits():
    """launch_dependent only ever takes kernels that call dependency_wait()."""
    kernels = {f[1]: f[3] for f in functions() if f[0] == "global"}
    names = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        names |= set(re.findall(r"launch_dependent\((\w+_kernel)", open(path).read()))
    assert names and all("dependency_wait()" in kernels[n] for n in names), names


def test_flags_that_blocks_branch_on_are_constant():
    """A kernel whose blocks leave early on a matrix's ok flag does not write it:
    another block of the same matrix may be reading it then, and threads of one
    block that read different values would part before a barrier. (The kernel
    that closes a chunk has one warp per matrix, which reads before it writes.)"""
    kernels = {f[1]: f[3] for f in functions() if f[0] == "global"}
    leave = [k for k, b in kernels.items() if re.search(r"if \([^;{]*P\.ok\[b\] == 0[^;{]*\) return;", b)]
    assert "terms_delta_kernel" in leave and "terms_series_kernel" in leave
    for k in leave:
        assert not re.search(r"P\.ok\[[^]]*\]\s*=[^=]", kernels[k]), k


def test_side_streams_are_joined_before_the_scratch_is_freed():
    """Also on errors: after the launches' block and ahead of scratch_free, which
    frees in the order of the caller's stream alone."""
    s = open(os.path.join(CSRC, "api.cu")).read()
    body = s[s.index("int run_batch("):]
    lanes = re.search(r"SideWork ([\w, ]+);", body).group(1).split(", ")
    end = body[body.index("} while (0);"):]
    end = end[:end.index("scratch_free(dmem")]
    assert len(lanes) == 2 and all(re.search(r"^  %s\.join\(\);" % v, end, re.M) for v in lanes), lanes
