"""The per-launch timing records name the kernel that ran: every name given to a launch is a kernel of the file that launches it (or that
name and a suffix for what it is used for; a record over two stages has the name they share)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_18239_b200", "csrc")
# uses of the small dense product (k_rows_times_w), named by the entry points that call it
STEPS = {"k_head_lsw", "k_ctx_first"}


def _kernels(text):
    """Names of the kernels a source defines."""
    names = set()
    for m in re.finditer(r"__global__\s+void\s+", text):
        rest = re.sub(r"^__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*", "", text[m.end():m.end() + 400])
        names.add(re.match(r"(\w+)\s*\(", rest).group(1))
    return names


def test_launches_report_under_the_name_of_their_kernel():
    sources = {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu"))}
    kernels = {f: _kernels(t) for f, t in sources.items()}
    everywhere = set().union(*kernels.values())
    assert "k_score_tc" in kernels["k_score_tc.cu"] and "k_link_attn_tmem_tc" in kernels["k_link_attn_tmem_tc.cu"]
    wrong = []
    for f, text in sources.items():
        known = everywhere | STEPS if f == "lime_api.cu" else kernels[f]
        for name in re.findall(r'"(k_\w+)"', text):
            if not any(name == k or name.startswith(k + "_") or k.startswith(name + "_stage") for k in known):
                wrong.append((f, name))
    assert not wrong, wrong
