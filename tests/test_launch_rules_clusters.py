"""The dependent-launch rules for kernels launched by every helper of csrc/kernels.h.

test_launch_rules.py collects the kernels of `launch_dep(`; the decode kernel is
launched as clusters by `launch_dep_clusters(`.  Here every helper that sets
programmatic stream serialisation is found in kernels.h itself, and the kernels
they launch must keep the same rules: wait first, then trigger or return."""
import re

from test_launch_rules import _kernel_body, _sources, _strip_comments


def _helpers(src):
    """Names of the launch helpers: functions whose body sets the serialisation attribute."""
    out = set()
    for m in re.finditer(r"cudaError_t (\w+)\(void \(\*kernel\)", src):
        i = src.index("{", m.end())
        depth = 0
        for j in range(i, len(src)):
            depth += {"{": 1, "}": -1}.get(src[j], 0)
            if depth == 0:
                break
        if "ProgrammaticStreamSerialization" in src[i:j]:
            out.add(m.group(1))
    return out


def _launched(srcs, helpers):
    names, calls = set(), 0
    for f, s in srcs.items():
        if f == "kernels.h":
            continue
        calls += len(re.findall(r"\b(?:%s)\(" % "|".join(helpers), s))
        for m in re.finditer(r"\b(?:%s)\(\s*([A-Za-z_][\w:]*)" % "|".join(helpers), s):
            names.add(m.group(1).split("::")[-1])
    return names, calls


def check(body, name):
    w = body.find("dep_wait()")
    assert w >= 0, "%s never calls dep_wait()" % name
    launch = body.find("dep_launch()")
    assert launch < 0 or launch > w, "%s calls dep_launch() before dep_wait()" % name
    assert re.search(r"\breturn\b", body[:w]) is None, "%s may return before dep_wait()" % name


def test_every_dependent_kernel_keeps_the_rules():
    srcs = {f: _strip_comments(s) for f, s in _sources().items()}
    helpers = _helpers(srcs["kernels.h"])
    assert {"launch_dep", "launch_dep_clusters"} <= helpers
    names, _ = _launched(srcs, helpers)
    assert {"decode_tiles_kernel", "decode_merge_kernel", "compact_kernel", "threshold_kernel", "lse_merge_kernel",
            "score_lse_tc_kernel", "score_colsum_tc_kernel", "fuse_v_tcp_kernel"} <= names, names
    for name in sorted(names):
        bodies = [b for b in (_kernel_body(s, name) for s in srcs.values()) if b is not None]
        assert len(bodies) == 1, "%s: a launch helper's argument is not a kernel's own name" % name
        check(bodies[0], name)


def test_decode_reads_and_writes_nothing_before_the_wait():
    # the one dependent kernel that follows arbitrary work: no access through its
    # pointer parameters before dep_wait()
    body = _kernel_body(_strip_comments(_sources()["decode.cu"]), "decode_tiles_kernel")
    head = body[:body.index("dep_wait()")]
    for p in ("q", "Kc", "Vc", "Kt", "Vt", "Kq", "Vq", "Kqp", "Vqp", "out", "part_o", "part_ml"):
        assert re.search(r"\b%s\b" % p, head) is None, p


def test_a_missing_wait_is_seen():
    body = _kernel_body(_strip_comments(_sources()["decode.cu"]), "decode_tiles_kernel")
    moved = body.replace("dep_wait();", "", 1)
    moved = moved.replace("dep_launch();", "dep_launch(); dep_wait();", 1)
    try:
        check(moved, "moved")
    except AssertionError:
        return
    raise AssertionError("a trigger before the wait was not seen")
