"""What no run can show: rules that the kernels' sources keep."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_02470_b200", "csrc")


def _instructions(name):
    text = "".join(open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))))
    return re.findall(name + r"[\w.:]*", text)


def test_hand_offs_between_ctas_release_at_cluster_scope():
    """An arrival on another CTA's barrier names its scope (the default is the CTA, which orders nothing between two of them): release
    behind shared memory, relaxed where tensor memory and its fences carry the data; and the wait that belongs to it does, too."""
    remote = [i for i in _instructions(r"mbarrier\.arrive") if "shared::cluster" in i]
    assert remote and all(".release.cluster." in i or ".relaxed.cluster." in i for i in remote), remote
    waits = _instructions(r"mbarrier\.try_wait")
    assert any(".acquire.cluster." in i for i in waits) and any(".relaxed.cluster." in i for i in waits)


def test_votes_do_not_stand_in_for_warp_barriers():
    """A vote orders no memory: where lanes read what others wrote to shared memory before a wait that ends in one, a __syncwarp follows."""
    text = open(os.path.join(CSRC, "eig_tridiag.cu")).read()
    step = text[text.index("auto step = [&]"):text.index("// both vectors at this thread's columns")]
    assert re.search(r"wait_bytes\([^;]*\)\) return [^;]*;\s*__syncwarp\(\);", step)


def test_the_first_static_selection_loads_every_kernel_of_the_others():
    """sage_select_static promises that no call but the first on a device loads anything, whatever the sizes: every kernel that the
    launchers behind it name is in the list that the first call goes through."""
    text = open(os.path.join(CSRC, "select.cu")).read()

    def body(name):
        at = re.search(r"\n[^\n]*\b" + name + r"\([^;{]*\{", text)
        return text[at.start():text.index("\n}\n", at.end())]

    used = set()
    for f in ("run_rank", "run_top_keys", "run_cluster_sort", "sort_launches"):
        used |= set(re.findall(r"launch(?:_chained)?\((k_\w+)", body(f))) | set(re.findall(r"\b(k_\w+)<<<", body(f)))
    assert used == set(re.findall(r"\(const void\*\)(k_\w+)", body("load_selection"))) and len(used) >= 7
