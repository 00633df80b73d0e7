"""Threads that use the library for the first time together, each with a context and a stream of its own, get what one thread
gets: a fresh process, since the library's kernels are set up once per process and device."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import threading
import torch
from paper_2503_07518_b200 import binding as tb

THREADS = 8

def inputs():
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.bfloat16)
    E, hid, n_tok = 1024, 512, 16
    predictor = [rand(n_tok, E), rand(E), rand(E), rand(hid, E) / 32, rand(1, 8, 32, hid) / 16]
    ctx = []
    for L in (12000, 700):                               # a cluster per list, a block per list
        c = tb.Context(1, 8, 2, 128, 32, tb.TB_BF16, 1, L, 500)
        c.set_projection(0, rand(2, 128, 32))
        c.append_kv(0, 1, None, [L], rand(L, 2, 128), rand(L, 2, 128))
        ctx.append(c)
    return predictor, ctx, rand(1, 1, 8, 128)

def work(predictor, ctx, q, out):
    hidden, ln_w, ln_b, w1, w2 = predictor
    q_imp = torch.empty(1, hidden.shape[0], 8, 32, device="cuda")
    scratch = torch.empty(hidden.shape[0], w1.shape[0], device="cuda")
    assert tb.TB_OK == tb.predict_importance_queries(hidden, ln_w, ln_b, w1, w2, tb.TB_BF16, 8, 1, 32, scratch, q_imp)
    out.append(q_imp)
    for c in ctx:
        L = c.get_length(0, 0)[0]
        c.project_keys(0, 1, None, [0], [L])
        idx = torch.zeros(1, 1, 2, c.index_capacity, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, 1, 2, dtype=torch.int32, device="cuda")
        o = torch.empty(1, 1, 8, 128, device="cuda")
        p = tb.select_params(400)
        c.select_topk(0, 1, None, 1, q_imp[:, :1].contiguous(), p, idx, cnt)
        c.sparse_decode_attention(0, 1, None, 1, q, p, o)
        assert c.get_status() == 0
        out += [idx, cnt, o]

state = [inputs() for _ in range(THREADS)]
results = [[] for _ in range(THREADS)]
errors = []
start = threading.Barrier(THREADS)

def run(i):
    try:
        with torch.cuda.stream(streams[i]):
            start.wait()
            work(*state[i], results[i])
            streams[i].synchronize()
    except BaseException as e:
        errors.append(repr(e))

streams = [torch.cuda.Stream() for _ in range(THREADS)]
torch.cuda.synchronize()
threads = [threading.Thread(target=run, args=(i,)) for i in range(THREADS)]
[t.start() for t in threads]
[t.join() for t in threads]
assert not errors, errors
alone = []
work(*state[0], alone)
torch.cuda.synchronize()
for r in results:
    assert len(r) == len(alone) and all(torch.equal(a, b) for a, b in zip(r, alone))
print("threads agree")
"""


def test_first_uses_by_several_threads():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "threads agree" in r.stdout, r.stdout + r.stderr
