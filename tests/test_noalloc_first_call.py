"""The allocation-free call takes nothing from the device once its first call is made, whatever sizes follow."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# (heads, queries, keys): whole pairs; equal pieces; more than sixteen of them; shares of a line
ROUTES = [(2, 300, 200), (8, 687, 2748), (1, 256, 4000), (15, 1280, 2432)]


def test_the_first_call_loads_every_kernel():
    from fake_cuda import FakeLibrary
    for first in range(len(ROUTES)):
        fake = FakeLibrary()
        for head_dim in (64, 128):
            for n, (heads, n_q, n_k) in enumerate([ROUTES[first]] + ROUTES):
                rc = fake.lib.headcast_dense_attend_noalloc(4096, 4096, 4096, 4096, n_q, n_k, heads, head_dim, 0.0, 11)
                assert rc == 0
                if n == 0 and head_dim == 64:
                    loaded = fake.kernels_loaded()
        assert fake.kernels_loaded() == loaded


def in_fresh_process(code):
    code = "import sys\nsys.path.insert(0, %r)\nimport torch\nfrom paper_2607_20125_b200 import binding\n" % ROOT + code
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT, timeout=300)
    assert res.returncode == 0, res.stdout + res.stderr


@pytest.mark.gpu
def test_free_memory_stays_the_same_after_the_first_call():
    in_fresh_process("""
routes = %r
sets = [[torch.zeros(n, h, d, dtype=torch.bfloat16, device="cuda") for n in (q, k, k, q)] for h, q, k in routes for d in (64, 128)]
binding.dense_attend_noalloc(*sets[0])
binding.noalloc_status()
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
for s in sets:
    binding.dense_attend_noalloc(*s)
binding.noalloc_status()
assert torch.cuda.mem_get_info()[0] == free, (free, torch.cuda.mem_get_info()[0])
""" % ROUTES)


@pytest.mark.gpu
def test_programs_that_make_no_such_call_do_not_hold_its_scratch():
    in_fresh_process("""
q = torch.zeros(48, 4, 64, dtype=torch.bfloat16, device="cuda")
out = torch.empty_like(q)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
hc = binding.HeadCast(4, 64, 4, 4, 2)
hc.append(q, q)
hc.full_attend(q, out)
hc.append(q, q)
hc.classify(q)
hc.split_cache()
hc.attend(q, out)
hc.check()
hc.destroy()
binding.release_memory()
assert free - torch.cuda.mem_get_info()[0] < 16 << 20  # what is left is the kernels' code
""")
