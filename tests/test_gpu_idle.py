"""The loop leaves the GPU by itself when nothing comes, any number of times."""
import time

import numpy as np
import pytest
import torch

from paper_2604_07609_b200 import binding as B
from synth import make_weights
from synth.configs import ModelCfg, SchedCfg

pytestmark = pytest.mark.gpu


def test_many_idle_exits_in_a_row():
    """Every exit is a decision that all warps of the control CTA have to take together; when each had a clock of its own
    about one exit in a hundred never ended."""
    model = ModelCfg(1, 256, 8, 2, 64, 256, 512)    # four query heads per kv head: launched as CTA pairs
    sched = SchedCfg(max_batch=2, prefill_chunk_tokens=16, n_slots=4, max_prompt=8, max_new=2, n_blocks=8)
    w = make_weights(model, 3, "cpu").cuda()
    kv = torch.zeros(sched.n_blocks * B.kv_bytes_per_block(model, sched.block_size), dtype=torch.uint8, device="cuda")
    eng = B.Blink(model, sched, w, kv, idle_exit_us=200)
    try:
        n = 600
        for i in range(n):
            eng.blink_submit(np.array([1, 2, 3], np.int32), 1)
            assert len(eng.drain(1, timeout_s=20)) == 1
            t0 = time.monotonic()
            while eng.blink_get_stats().loop_state == B.LOOP_RUNNING:
                assert time.monotonic() - t0 < 10, f"exit {i} does not end"
        st = eng.blink_get_stats()
        assert st.loop_state == B.LOOP_EXIT_IDLE and st.device_status == 0 and st.launches >= n
    finally:
        assert eng.blink_destroy() == B.BLINK_OK


def test_phase_times_of_every_step_hold_its_last_phase():
    """One thread adds a phase's time, other lanes copy the array: with no order between the two the last phase of a step,
    sampling, could miss."""
    model = ModelCfg(1, 256, 8, 2, 64, 256, 512)
    sched = SchedCfg(max_batch=2, prefill_chunk_tokens=16, n_slots=4, max_prompt=8, max_new=500, n_blocks=80)
    kv = torch.zeros(sched.n_blocks * B.kv_bytes_per_block(model, sched.block_size), dtype=torch.uint8, device="cuda")
    eng = B.Blink(model, sched, make_weights(model, 3, "cpu").cuda(), kv, exec_mode=B.EXEC_MANUAL, stats_iters=1024)
    try:
        eng.blink_submit(np.array([1, 2, 3], np.int32), 500)
        eng.blink_run(499)
        its = eng.blink_get_iter_stats()
        assert len(its) == 499
        phases = its["phase_ns"].astype(np.int64)
        assert (phases[:, 11] > 0).all()          # one phase in rows this short: its time is there or it is not
        # no more than the time between control plane and post step (the rest is the first barrier and the step's set-up)
        assert (phases.sum(axis=1) <= (its["t_end_ns"] - its["t_forward_ns"]).astype(np.int64)).all()
    finally:
        assert eng.blink_destroy() == B.BLINK_OK
