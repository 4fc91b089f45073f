"""First builds of banks of many geometries from several host threads at once:
the kernels' shared-memory limits are raised on first use, and one thread's
smaller one must not undercut the other's launch."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import threading
import torch
import paper_1711_01177_gb300 as grim, synth
N, THREADS, ROUNDS = 20_000, 8, 60
r2 = torch.from_numpy(synth.pack2bit(synth.ref_iid(N, 3))).cuda()
failed = []
gate = threading.Barrier(THREADS)
def builds(which):
    try:
        stream = torch.cuda.Stream()
        for i in range(ROUNDS):
            gate.wait(60)
            # every length is the longest so far, by a few bases more or less
            bank = grim.grim_build_bank(r2, N, 5, 17 + 2 * (THREADS * i + which), 100, stream=stream)
            gate.wait(60)
            for _ in range(3):  # and once more with the limit as the threads left it
                grim.grim_build_bank_into(bank, r2, stream=stream)
            stream.synchronize()
            bank.free()
    except Exception as e:
        failed.append(repr(e))
        gate.abort()
threads = [threading.Thread(target=builds, args=(w,)) for w in range(THREADS)]
[t.start() for t in threads]
[t.join() for t in threads]
assert not failed, failed
"""


def test_threads_build_first_banks_of_many_sizes():
    import paper_1711_01177_gb300 as grim
    grim.build()
    for _ in range(4):  # the limits are set once a process
        r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
