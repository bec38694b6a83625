"""Kernels that start before the stream's previous kernel has ended (grid_sync() in their body) must
read what that kernel writes with plain loads: the read-only path (__ldg, const __restrict__) is for
data that does not change while the kernel lives, and the compiler may move such a load above the
wait.  On that path may be only the tables that set-up calls wrote several kernels before (twiddles,
Box-Muller, multipliers, the sqrt(P) field), and the inputs of kernels whose launch is not overlapped:
the shell weights of X_PKADJ, g_S (g0) of k_z_adj_source_cta, and all of k_cic_grad's."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1909_06282_gb300", "csrc")
TABLES = {"g_tab", "a.mt0", "a.mt1", "mp", "a.scf", "sp"}


def sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def test_read_only_loads_are_of_tables():
    src = sources()
    # k_cic_grad and the gather that only it calls: an ordinary launch
    p, m = src["passes.cuh"], src["misc.cu"]
    assert m.count("cic_gather_grad<N>(") == 1 and "cic_gather_grad<N>(" not in p
    grad = m[m.index("k_cic_grad(CicGradArgs a)"):m.index("cudaError_t launch_cic_grad_n(")]
    gather = p[p.index("void cic_gather_grad("):p.index("// Transpose of k_z_source.")]
    assert "cic_gather_grad<N>(" in grad and m.count("k_cic_grad<N><<<") == 1 and "launch_overlapped(k_cic_grad" not in m
    src["misc.cu"], src["passes.cuh"] = m.replace(grad, ""), p.replace(gather, "")
    seen = set()
    for text in src.values():
        seen |= {m.group(1) for m in re.finditer(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?([\w.]+)", text)}
    assert seen <= TABLES | {"a.shell_w", "g0"}
    # the weights are read in X_PKADJ only, and its launch is an ordinary one
    p = src["passes.cuh"]
    assert p.count("__ldg(a.shell_w") == 1
    launch = p[p.index("cudaError_t launch_x_m("):p.index("cudaError_t launch_x_t(")]
    assert re.search(r"if constexpr \(MODE == X_PKADJ\) \{[^}]*k<<<[^}]*return cudaGetLastError\(\);\s*\}", launch)
    cta = p[p.index("k_z_adj_source_cta(ZAdjSourceArgs a)"):p.index("k_z_adj_source_fp(ZAdjSourceArgs a)")]
    assert p.count("__ldg(g0") == cta.count("__ldg(g0")
    assert p.count("(k_z_adj_source_cta<N>, a, s, false)") == p.count("k_z_adj_source_cta<N>")
    assert re.search(r"if \(!overlap\) \{[^}]*k<<<[^}]*return cudaGetLastError\(\);\s*\}", p)


def test_overlapped_kernels_take_no_restricted_inputs():
    for f, text in sources().items():
        for m in re.finditer(r"__global__[^;{]*\{", text):
            end = text.find("\n}\n", m.start())
            if "grid_sync()" in text[m.start():end]:
                assert "__restrict__" not in m.group(0), (f, m.group(0))
    # functions inlined into them: restricted inputs are the tables
    for f in ("passes.cuh", "fft_core.cuh", "boxmuller.cuh"):
        for name in re.findall(r"const \w+\s*\*\s*__restrict__ (\w+)", sources()[f]):
            assert name in {"tw", "g_tw", "g_tab"}, (f, name)
