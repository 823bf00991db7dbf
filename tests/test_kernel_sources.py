"""Rules of the kernel sources that no run can show reliably, checked on the
text: a kernel that is launched to start while its predecessor still runs
(launch_after, grid_start) reads what that predecessor writes, so those reads
may not take the read-only path, which supposes data that nothing writes while
the kernel runs."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_03857_gb300", "csrc")
# the files whose device code runs inside kernels launched by launch_after
OVERLAPPED = ("lb_common.cuh", "lb_cell.cuh", "lb_march.cuh", "lb_tile.cuh", "lb_forms.cuh", "lb_step3.cu",
              "lb_step_rec.cu", "lb_step_batch.cu", "lb_rev_tile.cuh")


def source(name):
    """The file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def calls(text, name):
    """The argument lists of every call of `name` in text."""
    out = []
    for m in re.finditer(r"\b%s\s*(<[^<>()]*>)?\(" % name, text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        out.append((m.group(1) or "", text[m.end():i - 1].strip()))
    return out


def test_every_overlapped_kernel_file_is_listed():
    using = {os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu*"))
             if re.search(r"\b(grid_start|launch_after)\s*\(", source(os.path.basename(p)))}
    assert using - set(OVERLAPPED) == {"lb_adjoint.cu"}  # (its rev_tile is in lb_rev_tile.cuh)


def test_overlapped_kernels_read_written_data_coherently():
    """Read-only loads there: theta_b and a batch's tables, which only copies
    write, and copies are never overlapped. The state loads (lb_ld) are of one
    kind, and no pointer is promised to be unaliased."""
    allowed = ("P.thb", "tiles +", "reinterpret_cast<const int*>(src)")
    for name in OVERLAPPED:
        text = source(name)
        for fn in ("__ldg", "lb_ldg"):
            for _, args in calls(text, fn):
                assert args.startswith(allowed), (name, fn, args)
        assert not calls(text, "lb_ld"), name
        for line in text.splitlines():
            if "__restrict__" in line:
                assert re.search(r"const (StepParams|int2)\* __restrict__ (src|table|tiles)\b", line), (name, line)
                assert "float" not in line.split("__restrict__")[0], (name, line)


def test_nothing_about_a_device_is_kept_for_the_process():
    """A shared-memory opt-in, an SM count or an occupancy looked up once per
    process would serve a second device's launches with the first one's."""
    for path in glob.glob(os.path.join(CSRC, "*.[ch]*")):
        for line in source(os.path.basename(path)).splitlines():
            assert not re.match(r"\s+(static|thread_local)\s+(?!constexpr|__device__)[^()]*=", line), (path, line)


def test_read_backs_run_on_their_own_device():
    """Read-backs and state copies were copies, which run wherever their
    memory is; as kernels they need their handle's device to be current."""
    text = source("lb_host.cu")
    seen = 0
    for m in re.finditer(r"\b(launch_collect|launch_copy_state)\(", text):
        scope = text.rfind("const OnDevice on(", 0, m.start())
        assert scope >= 0 and "\n}\n" not in text[scope:m.start()], text[m.start() - 200:m.start() + 40]
        seen += 1
    assert seen == 4
    asked = [args for _, args in calls(text, "on_device_memory") if not args.startswith("const void*")]
    assert len(asked) == 4 and all(a.endswith("h->dev") for a in asked)


def test_heat_flux_terms_go_through_the_checked_accesses():
    """The checked build sees every global access of the step: the columns'
    terms of q(t) too."""
    for name in OVERLAPPED:
        text = source(name)
        assert not re.search(r"\bP\.q(part|prev)\s*\[", text), name
        plain = [a for fn in ("__ldcg", "__ldg", "__stcg") for _, a in calls(text, fn) if "P.q" in a]
        assert not plain, (name, plain)
