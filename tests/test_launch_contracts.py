"""CPU: what the dependent launches (pdl.cuh) rest on, read from the kernels'
source.  Every kernel launched dependent waits for its predecessors and does
not promise the compiler that their outputs stay unchanged; one that
allocates tensor memory lets the next kernel start only after its block
holds its columns (a dependent that took them first could wait for its own
predecessor for ever).  The GPU case runs the shapes of which several blocks
share an SM (edges 18 to 48) from many contexts at once."""
import os
import re
import threading

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1406_0835_gb300", "csrc")


def sources():
    return {f: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
            for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def kernels():
    """name -> (parameters, body) of every __global__ function."""
    out = {}
    for text in sources().values():
        for m in re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\(([^{;]*)\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out[m.group(1)] = (m.group(2), text[m.end():i])
    return out


def dependent():
    names = set()
    for text in sources().values():
        names |= set(re.findall(r"pdl_launch\(\s*(k_\w+)", text))
    return names


def test_dependent_kernels_wait():
    k, d = kernels(), dependent()
    assert len(d) > 30
    for name in sorted(d):
        assert re.search(r"\bpdl_(wait|enter)\(\)", k[name][1]), name


def test_tensor_memory_is_held_before_the_next_kernel_may_start():
    k, d = kernels(), dependent()
    holders = [n for n in d if "tmem_alloc" in k[n][1]]
    assert sorted(holders) == ["k_force", "k_tline"]
    for n in holders:
        body = k[n][1]
        assert "pdl_enter" not in body, n
        assert body.count("pdl_trigger()") == 1, n
        # the allocating warp's barrier lies between the two
        known = re.search(r"bar_arrive\(4,.*?bar_sync\(4,|__syncthreads\(\)", body[body.index("tmem_alloc"):], re.S)
        assert body.index("tmem_alloc") + known.end() < body.index("pdl_trigger()"), n
        assert body.index("pdl_wait()") < body.index("pdl_trigger()"), n


def test_dependent_kernels_restrict_only_tables():
    """A __restrict__ parameter tells the compiler that nothing changes what it
    points to while the kernel runs, so that its loads need not stay behind the
    wait; only the functional's table, written at set-up, may be one."""
    k = kernels()
    for name in sorted(dependent()):
        assert set(re.findall(r"__restrict__\s+(\w+)", k[name][0])) <= {"tab"}, name


def test_the_static_entry_waits_for_its_tables():
    """A copy from pageable memory may return before the data have arrived, and
    the caller's stream need not follow the default stream: the one-time
    uploads run on the caller's stream and are waited for."""
    text = sources()["capi_static.cu"]
    setup = text[text.index("device_setup("):text.index("d.ready = true")]
    assert "cudaMemcpy(" not in setup
    copies = re.findall(r"cudaMemcpyHostToDevice, (\w+)\)", setup)
    assert copies == ["st", "st"]
    assert setup.index("cudaStreamSynchronize(st)") > setup.rindex("cudaMemcpyAsync")


def test_a_wait_that_runs_out_is_flagged_before_its_products_are_committed():
    """k_tline's readers look at s_bad once a unit's products are done, so the
    issuing warp has to have raised it before it commits them."""
    text = sources()["kernels_tline.cu"]
    body = text[text.index("void issue("):text.index("store_lines(")]
    waits = re.findall(r"[^;{}]*mbar_wait\([^;]*", body)
    assert len(waits) == 1 and waits[0].strip().startswith("if (!tc::mbar_wait(bar, 0))")
    raised = body.index("*bad = 1;")
    assert raised < body.index("__threadfence_block()", raised) < body.index("mma_commit")
    assert re.search(r"wait\(full[^;]*;.*mma_commit", body, re.S)


FIRST_CALL = """
import numpy as np, torch
from paper_1406_0835_gb300 import inputs, ofdft
d = inputs.hydrogen(8, 1.0, 1.0e5, (24, 20, 30), seed=3, functional="vt84f")
N = 24 * 20 * 30
p = torch.full((N,), float(np.sqrt(8.0 / np.prod(d["L"]))), dtype=torch.float64, device="cuda")
p *= 1.0 + 0.1 * torch.cos(torch.arange(N, device="cuda", dtype=torch.float64))
torch.cuda.synchronize()
s, out = torch.cuda.Stream(), []
for _ in range(2):
    v = torch.zeros_like(p)
    torch.cuda.synchronize()
    E = ofdft.ofdft_energy_potential_static(np.diag(d["L"]), d["grid"], d["ions"], d["Z"], d["T"], "vt84f",
                                            p.data_ptr(), v.data_ptr(), stream=s.cuda_stream)
    out.append((E["F_tot"], v.cpu().numpy()))
assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1]) and np.all(out[0][1] != 0.0)
"""


@pytest.mark.gpu
def test_first_static_call_on_a_non_blocking_stream():
    """In a process of its own; the second call repeats the first bit for bit."""
    import subprocess
    import sys
    import __graft_entry__
    __graft_entry__.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", FIRST_CALL], cwd=root, check=True, timeout=600)


@pytest.mark.gpu
def test_small_edges_of_many_contexts_share_the_sms():
    """Eight contexts minimise at once from eight threads, edges of 128 and of
    256 columns mixed; each result repeats its solo run bit for bit."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_1406_0835_gb300 import inputs, ofdft
    grids = [(18, 32, 128), (32, 30, 96), (24, 48, 60), (32, 32, 32), (30, 64, 32), (20, 24, 120), (48, 50, 18), (32, 20, 144)]
    ctxs = []
    for i, grid in enumerate(grids):
        d = inputs.hydrogen(8, 1.0, 1.0e5, grid, seed=i, functional="vt84f")
        ctxs.append(ofdft.Context(d["L"], grid, d["ions"], d["Z"], d["T"], "vt84f"))
    solo, both = [], [None] * len(ctxs)
    for c in ctxs:
        c.set_phi()
        solo.append(c.minimize(gtol=1e-6)[0]["F_tot"])

    def work(i):
        ctxs[i].set_phi()
        both[i] = ctxs[i].minimize(gtol=1e-6)[0]["F_tot"]
    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(ctxs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for c in ctxs:
        c.close()
    assert np.array_equal(solo, both)
