"""Closing the server while every slot is busy and requests still wait: the scheduler
waits for a slot (no spinning) and serves them all."""
import time

import torch

from paper_1410_0260_gb300.serve import Request, Server
from test_serving_host import _Tree


def test_close_serves_what_waits_without_spinning():
    tree = _Tree()
    srv = Server(tree, torch.ones((tree.N, 1)), n_slots=1, budget_bytes=10 ** 9, max_cols=16)
    ctx = srv.slots[0].ctx
    slow = ctx.evaluate
    ctx.evaluate = lambda stream=None: (time.sleep(0.3), slow(stream))[1]
    reqs = [srv.submit(Request("weights", torch.ones((tree.N, 16)))) for _ in range(3)]
    while not srv.slots[0].busy:
        time.sleep(0.001)
    cpu = time.process_time()
    srv.close()
    cpu = time.process_time() - cpu
    assert all(r.done.is_set() and r.error is None for r in reqs)
    assert cpu < 0.3                     # of about 0.9 s asleep in the evaluations
