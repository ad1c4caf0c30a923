"""Distributed shared memory may be touched once every block of the cluster is known to have started, so in every kernel a
cluster barrier's wait stands in front of the first remote access.  What goes wrong without it depends on when blocks start
and cannot be provoked on purpose, so the order is checked in the sources, on the CPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_16626_b200", "csrc")
REMOTE = ("st.shared::cluster", "st_cluster_v4(", "st_cluster_u32(", "mbar_arrive_remote(", "atom.shared::cluster", "red.shared::cluster", "ld.shared::cluster",
          "st_async_v4(", "ld_cluster_f32(", "ld_cluster_u32(")
WAIT = ("barrier.cluster.wait", "cluster_wait()", "cluster_sync_all()")


def kernels():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for piece in re.split(r"(?=__global__ void)", text)[1:]:
            body = piece[:piece.find("\n}\n")]
            name = re.search(r"(\w+)\s*\(const|(\w+)\s*\(int|(\w+_kernel)\s*\(", body)
            if any(t in body for t in REMOTE):
                found.append(((name.group(1) or name.group(2) or name.group(3)) if name else "?", body))
    return found


def test_there_are_such_kernels():
    names = [n for n, _ in kernels()]
    assert {"hif8_gemm_warp_kernel", "hif8_gemm_narrow_kernel", "hif8_gemm_weights_kernel", "bf16_gemm_pair_kernel"} < set(names), names


def test_every_remote_access_is_known_here():
    # helpers that touch another block's shared memory are called from kernels by a name in the list above
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for name, code in re.findall(r"__device__ __forceinline__ \w+ (\w+)\([^)]*\)\s*\{(.*?)\n\}", text, flags=re.S):
            if re.search(r'"(st|ld|atom|red|mbarrier\.arrive)[\w.]*\.shared::cluster', code):
                assert name + "(" in REMOTE, (path, name)


@pytest.mark.parametrize("name,body", [pytest.param(n, b, id=n) for n, b in kernels()])
def test_remote_accesses_follow_a_cluster_barrier(name, body):
    first_remote = min(body.find(t) for t in REMOTE if t in body)
    first_wait = min((body.find(t) for t in WAIT if t in body), default=-1)
    assert 0 <= first_wait < first_remote, name
