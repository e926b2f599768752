"""Kernels that overlap the ones before them (programmatic stream serialization): the
first statement of every kernel is the wait, and a kernel that is launched chained
promises constancy (`__restrict__`, __ldg, ld.global.nc) only of memory that no other
grid of the call writes.  Checked in the sources, as a broken promise need not show in
results."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_02510_gb300", "csrc")

# per chained kernel, the parameters that were complete before the call's last plain launch (the caller's
# inputs, results of an earlier call) or that no other grid of the call touches (the caller's outputs)
SETTLED = {
    "k_pr_seen": {"seen", "z"}, "k_pr_wkey": {"w_max"}, "k_pr_bin": {"seen", "z"},
    "k_sd_flags": {"seen", "pm", "z"}, "k_sd_priority": {"geom", "level", "delta", "z", "u"}, "k_sd_select": {"pm"},
    "k_sd_write": {"geom", "level", "dens", "sh"}, "k_ip_tail": {"holes"},
    "k_vx_hash": {"geom"},
    "k_lf_sobel": {"gt"}, "k_lf_loss": {"rgb", "gt", "w", "grad"}, "k_lf_loss4": {"rgb", "gt", "w", "grad"},
    "k_adam_flat": {"p", "grad", "m4", "v4"}, "k_adam_tail": {"p", "grad", "m", "v"},
    "k_emit": {"geom", "dens", "sh", "vidx"},
    "k_sh_bwd": {"rec", "cnt", "slot"},
    "k_debug_pairs": {"slot_vox", "s_dkey"},
    "k_render_f64": {"slot_vox", "geom", "dens", "sh", "pixels", "vidx", "rgb_out", "T_out"},
    "k_render_f64_rest": {"pixels", "rgb_out", "T_out"},
}
# helpers whose non-coherent loads read the caller's voxel arrays
NC_HELPERS = {"ld_row32", "sh_raw_row", "load_corners", "write_children"}


def text():
    out = ""
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        out += open(p).read()
    return re.sub(r"//[^\n]*", "", out)


def closing(s, i, pair):
    d = 1
    while d:
        d += (s[i] == pair[0]) - (s[i] == pair[1])
        i += 1
    return i


def kernels():
    """(name, parameter text, body text) of every __global__ function."""
    s = text()
    for m in re.finditer(r"__global__\s+void\s+", s):
        i = m.end()
        lb = re.match(r"__launch_bounds__\(", s[i:])
        if lb:
            i = closing(s, i + lb.end(), "()")
        name = re.match(r"\s*(\w+)", s[i:])
        i += name.end()
        i += re.match(r"\s*(<\w+>)?\s*\(", s[i:]).end()
        j = closing(s, i, "()")
        k = s.index("{", j) + 1
        yield name.group(1), s[i:j - 1], s[k:closing(s, k, "{}")]


def chained():
    return set(re.findall(r"\bchain\((k_\w+)", text()))


def test_sources_parse():
    names = {n for n, _, _ in kernels()}
    assert len(names) > 40 and chained() <= names and len(chained()) > 20


def test_every_kernel_waits_first():
    for name, _, body in kernels():
        assert re.match(r"\s*(grid_begin|grid_wait)\(\);", body), name


@pytest.mark.parametrize("name", sorted(chained()))
def test_chained_kernels_promise_only_settled_memory(name):
    for n, params, _ in kernels():
        if n == name:
            said = set(re.findall(r"__restrict__\s+(\w+)", params))
            assert said <= SETTLED.get(name, set()), said - SETTLED.get(name, set())


def test_non_coherent_loads_stay_in_the_named_helpers():
    s = text()
    for m in re.finditer(r"__ldg\(|\.nc\.", s):
        heads = list(re.finditer(r"__(?:device|global)__[^;{}()]*?\b(\w+)\s*\(", s[:m.start()]))
        assert heads[-1].group(1) in NC_HELPERS, s[m.start() - 80:m.end() + 40]


def test_nothing_in_a_walk_or_list_is_restrict():
    s = text()
    for m in re.finditer(r"\bstruct\s+\w+\s*\{", s):
        body = s[m.end():closing(s, m.end(), "{}")]
        fields = [f for f in re.findall(r"__restrict__\s+(\w+)\s*;", body)]
        assert not fields, fields


def test_no_two_grids_of_a_stream_wait():
    """grid_begin lets the next grid in only after its own wait: else every grid behind a slow one becomes
    resident, and their waiting blocks keep other streams' kernels out."""
    s = text()
    m = re.search(r"void grid_begin\(\)\s*\{([^}]*)\}", s)
    assert 0 <= m.group(1).find("grid_wait()") < m.group(1).find("launch_dependents")


def test_kernels_that_fill_the_gpu_let_no_grid_wait():
    """The LF steps run beside a forward: a grid waiting behind one of them would hold what that needs."""
    for name, _, body in kernels():
        if name in ("k_lf_sobel", "k_lf_digit", "k_lf_weight", "k_lf_loss", "k_lf_loss4", "k_fwd", "k_bwd"):
            assert re.match(r"\s*grid_wait\(\);", body), name
