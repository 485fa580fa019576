"""Rules of order that the kernels rely on and that no result shows while they are broken, checked in the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_01380_b200", "csrc")


def _kernels(name):
    """{kernel: body} of a source file, comments removed."""
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"//[^\n]*", "", text)
    out = {}
    for m in re.finditer(r"__global__\s+void\b", text):
        i = text.index("{", m.end())
        head, depth, j = text[m.end():i], 0, i
        while True:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
            if depth == 0:
                break
        out[re.search(r"\b(k_\w+)\s*\(", head).group(1)] = text[i:j]
    return out


def test_cluster_pieces_are_read_before_their_cta_may_leave():
    """The states of k_attn_own's pieces are read from peers' shared memory, and the barrier behind that orders nothing: every value
    that is read has to go into a result that is stored, or the read may be under way when the peer leaves.  So rows without a
    result read nothing.  The state starts where 16-byte words may: at the rounded base."""
    body = _kernels("nfd_attn_tc.cuh")["k_attn_own"]
    reads = [m.start() for m in re.finditer(r"ld_cluster_f[24]\(", body)]
    guard = body.rindex("if (w0.nsplit > 1", 0, min(reads))
    condition = body[guard:body.index("{", guard)]
    assert "w0.qt * 128 + trow < D.T" in condition and "16 * cq < D.dh" in condition
    assert body.index("attn_write<16>(", max(reads)) < body.index("cluster_", max(reads) + 40)
    assert re.search(r"state = reinterpret_cast<float \*>\(sh\.base \+ A::STATE_AT\)", body)


def test_marks_of_the_timeline_may_be_taken_in_functions():
    """The timeline's marks (builds with -DNFD_TRACE) are taken in functions that a kernel calls as well: their array belongs
    to the file and not to the kernel that opens its record, or such a build does not compile."""
    common = open(os.path.join(CSRC, "nfd_common.cuh")).read()
    t0 = re.search(r"#define NFD_TRACE_T0\(\)((?:[^\n]*\\\n)*[^\n]*)", common).group(1)
    assert "nfd_marks_" in t0 and "__shared__" not in t0
    assert re.search(r"^__shared__ unsigned long long nfd_marks_\[", common, re.M)


def test_plans_go_by_the_device_and_not_by_one_machine():
    """The number of SMs that a context's launches go by is asked of the device, in fp32 contexts too, and has no default that could
    pass for one."""
    text = open(os.path.join(CSRC, "nfd_fast.cuh")).read()
    assert re.search(r"int n_sm = 0\b", text)
    create = text[text.index("static int fast_create("):]
    assert create.index("cudaDevAttrMultiProcessorCount") < create.index("if (!bf16_mode) return")


def test_the_descriptor_and_the_modulation_are_complete_when_a_projection_starts():
    """The projections read both before their grid wait.  So the descriptor's writer releases nobody early, and every kernel up to
    the first projection of a pass waits before it releases its dependents."""
    kernels = _kernels("nfd_kernels.cuh")
    assert "pdl_launch()" not in kernels["k_set_params"]
    for name in ("k_temb", "k_gemv", "k_modw", "k_patch_embed", "k_adaln"):
        body = kernels[name]
        assert body.count("pdl_wait()") == body.count("pdl_launch()") == 1, name
        assert body.index("pdl_wait()") < body.index("pdl_launch()"), name
        # nobody leaves, and with it releases its dependents, before the wait
        assert "return" not in body[:body.index("pdl_wait()")], name
