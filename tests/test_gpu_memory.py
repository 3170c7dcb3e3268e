"""Device memory of preparation and of a handle's plan (GPU): the peak that
preparation reserves, and calls that still run when only the smaller of two forms
fits. Each case runs in a process of its own, whose memory pool starts empty."""
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

HEAD = """
import ctypes, math, sys
import torch
import paper_2009_12457_gb300 as bb

def complete(n, upward):
    # rows in descending order: unsorted on purpose
    v = torch.arange(n - 1, -1, -1, dtype=torch.int32, device="cuda")
    keep = v[None, :] > v.flip(0)[:, None] if upward else v[None, :] != v.flip(0)[:, None]
    ci = v[None, :].expand(n, n)[keep]
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = keep.sum(1).cumsum(0)
    torch.cuda.synchronize()
    return n, rp, ci

def leave(room):
    # takes device memory until the library can use `room` bytes
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    held = torch.empty(free - room, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    return held

def trim():
    # unused bytes of the library's block cache and pool go back to the driver
    bb.load()._ZN4bbtc21release_cached_blocksEiP11CUstream_st(0, None)
    rt, pool = ctypes.CDLL("libcudart.so.13"), ctypes.c_void_p()
    assert rt.cudaDeviceSynchronize() == 0
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert rt.cudaMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
"""


def run(body):
    proc = subprocess.run([sys.executable, "-c", HEAD + body], capture_output=True, text=True,
                          timeout=240)
    assert proc.returncode == 0, proc.stderr[-2000:]
    return proc.stdout.split()


def test_a_form_of_the_plan_that_fits_only_without_the_others():
    # 16 M in-edges: 128 MB as in-edges of all lists, 256 MB task by task
    got = run("""
import numpy as np
g = bb.Graph(*complete(5657, upward=True))
tasks = bb.bbtc_num_tasks(2)
ones = np.ones(tasks, dtype=np.uint8)
got = [math.comb(5657, 3), g.count(p=2), g.count(p=2, per_vertex=True)["total"]]
trim()
held = leave(200 << 20)
got.append(bb.bbtc_count(g.handle, bb.make_opts(p=2, task_mask=ones)))
got.append(g.count(p=2, per_vertex=True)["total"])
bb.bbtc_graph_plan(g.handle, bb.make_opts(p=2, task_mask=ones))
got.append(bb.bbtc_count(g.handle, bb.make_opts(p=2, task_mask=ones)))
out = g.count(p=2, per_vertex=True, per_task=True)
got += [int(out["per_task"].sum()), int(out["per_vertex"].sum()) // 3, g.count(p=2)]
print(*got)
""")
    assert len(got) == 9 and len(set(got)) == 1


@pytest.mark.parametrize("n", [4000, 16_400])
def test_symmetric_unsorted_rows_reserve_for_one_key_an_edge(n):
    # half of the entries give keys: by buckets up to 2^28 entries, beyond by sorting.
    # An entry's share: buckets 8 to 11 bytes or two sort buffers 8, distinct keys 4,
    # upward entries of the sorted attempt 4, columns and sources 4
    reserved, nnz, count, want = map(int, run(f"""
n, rp, ci = complete({n}, upward=False)
g = bb.Graph(n, rp, ci, symmetric=True)
print(bb.bbtc_device_memory()["pool_reserved"], ci.numel(), g.count(), math.comb(n, 3))
"""))
    assert count == want
    assert reserved < 24 * nnz


def test_general_input_that_only_fits_by_sorting():
    # 16 M entries: buckets of 268 MB, two sort buffers of 128 MB each
    count, want = map(int, run("""
n, rp, ci = complete(5657, upward=True)
held = leave(480 << 20)
h = bb.bbtc_graph_create(n, rp, ci)
del held
torch.cuda.empty_cache()
print(bb.bbtc_count(h), math.comb(n, 3))
"""))
    assert count == want
