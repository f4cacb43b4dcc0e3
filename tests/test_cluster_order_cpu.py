"""Order of the cluster kernels' accesses to one another's shared memory, read from their sources (no GPU): distributed
shared memory may be touched only once the CTA it belongs to is known to have started, i.e. behind a barrier over the
cluster, and every kernel of the library that touches it has such a barrier first."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_08134_b200", "csrc")
# what reaches into another CTA of the cluster, and what shows that it has started
REMOTE = ("st_cluster_u32", "ld_cluster_u32", "mbar_arrive_cluster", "bulk_copy_to_cta", "tma_load_2d_pair",
          "umma2_ss", "umma2_commit")
BARRIER = ("cluster_sync_all", "cluster_sync_relaxed", "cluster_wait")


def _block(text, at):
    """text[at] is '{': index just past its closing brace."""
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return i + 1
    raise AssertionError("unbalanced braces")


def _kernels():
    for fn in sorted(os.listdir(CSRC)):
        if not fn.endswith(".cu"):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, fn)).read())
        for m in re.finditer(r"__global__\s+void\b", text):
            params = text.index("(", text.index(")", m.end()) if "__launch_bounds__" in text[m.end():m.end() + 40] else m.end())
            name = re.findall(r"(\w+)\s*$", text[:params])[0]
            end = text.index("{", params)
            yield fn, name, text[end:_block(text, end)]


def _calls(body, names):
    return [m.start() for m in re.finditer(r"\b(?:%s)\s*\(" % "|".join(map(re.escape, names)), body)]


def _without_lambdas(body):
    """The body with its named lambdas blanked out, and the names of those that reach into another CTA."""
    reaching = []
    for m in list(re.finditer(r"auto\s+(\w+)\s*=\s*\[&\]", body)):
        start = body.index("{", m.end())
        end = _block(body, start)
        if _calls(body[start:end], REMOTE):
            reaching.append(m.group(1))
        body = body[:start] + " " * (end - start) + body[end:]
    return body, reaching


def test_every_kernel_passes_a_cluster_barrier_before_it_touches_another_cta():
    seen = []
    for fn, name, text in _kernels():
        body, reaching = _without_lambdas(text)
        remote = _calls(body, REMOTE + tuple(reaching))
        if not remote:
            continue
        barriers = _calls(body, BARRIER)
        assert barriers and min(barriers) < min(remote), f"{fn}: {name} touches another CTA before any cluster barrier"
        seen.append(name)
    assert {"gemm_tc_kernel", "gemm_persist_kernel", "swiglu_kernel", "attn_tc_kernel", "kth_cluster_kernel",
            "select_cluster_kernel"} <= set(seen), seen
