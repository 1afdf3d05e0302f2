"""Kernels that set the status word and synchronise their CTA take the decision whether to run once per CTA.  (The race
that separate reads by its warps would be cannot be provoked on a GPU without risking a hang, so the sources are read.)"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_11751_gb300", "csrc")
BARRIER = re.compile(r"__syncthreads|bar\.sync|ss_group_|prod_sync|tcgen05|chol_diag32|cluster_sync_all|_one_cta|item_rows")


def functions():
    """(file, name, body) of every kernel and of every item of the persistent kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"^(?:__global__|__device__ void item_)", text, flags=re.M):
            end = text.index("\n}", m.start())
            body = text[m.start():end]
            yield os.path.basename(path), re.search(r"\b(k_\w+|item_\w+)\s*\(", body).group(1), body


def test_status_is_taken_once_per_cta():
    seen, wrong = 0, []
    for path, name, body in functions():
        if "set_status(" not in body or not BARRIER.search(body):
            continue
        seen += 1
        # one thread's read that is shared through shared memory is one answer too; a cluster whose CTAs have all read the
        # status before any of them may set it needs nothing more
        rest = re.sub(r"if \(threadIdx\.x == 0\) \*go_s = load_status\(info\) == 0;", "", body)
        if "load_status(" in rest and not re.search(r"load_status\(info\) != 0\) return;\s*cluster_sync_all\(\);", rest):
            wrong.append(f"{path}: {name}")
    assert seen >= 14
    assert not wrong, wrong
