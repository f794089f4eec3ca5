"""Rules of the kernels that no run can show, checked on their source text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1004_5059_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def body_of(text, name):
    """The text between the braces of the function `name`."""
    at = text.index("{", re.search(r"%s\s*\([^;]*?\)\s*\{" % name, text).end() - 1)
    depth = 0
    for k in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[at:k + 1]
    raise AssertionError(name)


def test_a_network_kernel_that_gives_up_waits_for_its_copies_and_products():
    """A CTA must not exit with a bulk copy into its shared memory or a product in flight.  A barrier's
    wait for parity q returns at once while the phase in progress has the other parity, so the wait for
    the last of several loads on one barrier needs the parity of that load: it flips with every issue."""
    text = source("tvlbm_mlp.cu")
    train = body_of(text, "mlp_train_kernel")
    first, later = [m.end() for m in re.finditer(r"tma_load_2d\(xs, &mx, &x_bar, [^;]*;", train)]
    assert re.match(r"\s*xph \^= 1;", train[later:])
    assert train.count("xph ^= 1") == 1 and re.search(r"uint32_t xph = 0;", train)
    gave_up = train[train.index("atomicOr(status, 1)"):]
    assert re.search(r"bar_wait\(&w_bar, 0\);\s*bar_wait\(&x_bar, xph\);\s*mma_commit\(&end_bar\);\s*bar_wait\(&end_bar, 0\);", gave_up)
    forward = body_of(text, "mlp_fused_forward_kernel")
    gave_up = forward[forward.index("atomicOr(status, 1)"):]
    assert re.search(r"bar_wait\(&load_bar, 0\);\s*mma_commit\(&end_bar\);\s*bar_wait\(&end_bar, 0\);", gave_up)
    # the parity on a model of the barrier: load n completes phase n; a wait for parity q returns at once
    # unless the phase in progress has parity q
    for tiles in range(1, 6):
        for landed in (tiles - 1, tiles):  # all loads but the last, or all of them
            xph = (tiles - 1) & 1          # flipped with every load after the first
            returns_at_once = landed & 1 != xph
            assert returns_at_once == (landed == tiles)


def test_sweeps_that_overlap_load_populations_coherently():
    """A kernel launched with programmatic overlap begins before the kernel that writes its input has ended;
    a non-coherent load is only defined for data that does not change while the kernel runs."""
    text = source("tvlbm_kernels.cuh")
    codecs = text[text.index("ld_pop(const double"):text.index("split_rest")]
    assert "__ldg" not in codecs and ".nc" not in codecs
    assert len(re.findall(r"static R ld\(const T\* p\)", codecs)) == len(re.findall(r"struct Codec\w+ \{", codecs)) == 5
    # the others that read populations through __ldg are launched without overlap, every time
    for name, kernels in (("tvlbm_kernels_impl.cuh", ["sweep_lanes_kernel", "row_pop_means_kernel", "reencode_kernel"]),
                          ("tvlbm_fvlb.cu", ["fv_update64_kernel"]), ("tvlbm_mesh.cu", [])):
        text, rest = source(name), source(name)
        for kernel in kernels:
            launches = re.findall(r"(\w+)\((\w+),\s*%s\b|\b%s(?:<[^;()]*?>)?(<<<)" % (kernel, kernel), text)
            assert launches and all(l == ("launch_as", "false", "") or l[2] for l in launches), (kernel, launches)
            rest = rest.replace(body_of(text, kernel), "")
        # what remains are tables that the host wrote before the first launch
        for arg in re.findall(r"__ldg\(([^()]*)", rest):
            assert re.match(r"(src|wt|len|h|fp\.ysc) ?\+", arg), (name, arg)


def test_one_count_of_the_sms():
    """The lines between kernels and the splits of work use one SM count, with one fallback."""
    defined = [n for n in sorted(os.listdir(CSRC)) if re.search(r"\bint \w*sm_count\(\) \{", source(n))]
    assert defined == ["tvlbm_kernels.cuh"]


def test_activation_is_the_kernels_own():
    """tvlbm_mlp_activation runs the functions that the network's epilogues run, and there are no others."""
    text = source("tvlbm_mlp.cu")
    act = body_of(text, "activation_kernel")
    assert "gelu2_f(" in act and "gelu2_f(" in body_of(text, "mlp_fused_forward_kernel")
    assert "gelu2_both(" in act and "gelu2_both(" in body_of(text, "mlp_train_kernel")
    assert set(re.findall(r"\b(gelu\w*)\(", text)) == {"gelu2_f", "gelu2_both"}
