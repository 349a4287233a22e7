"""Servers of small requests keep as many workers on an SM as their blocks and slots allow
(needs a GB300)."""
import ctypes
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2002_11710_gb300 import _lib, api, gen, serve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,per_sm", [(128, 4), (256, 2), (512, 1)])
def test_workers_of_small_slots(threads, per_sm):
    """Slots of 40 missions, 8 vehicles and 30 locations take 22 KB by the full evaluation."""
    srv = serve.Server(max_loc=30, max_vehicles=8, max_missions=40, n_slots=64)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    insts = [gen.random_instance(60 + k, n_loc=30, n_vehicles=1 + k % 8, n_missions=1 + 3 * k % 40, duty_cap=500, max_minutes=90)
             for k in range(48)]
    srv.start(api.make_params(6, 80, gen.PENALTY, 1000, block_threads=threads), max_ctas=8 * sms)
    try:
        for k, i in enumerate(insts):
            assert srv.submit(i, k) is not None
        done, t0 = {}, time.perf_counter()
        while len(done) < len(insts):
            for slot, seq in srv.poll():
                done[seq] = srv.result(slot)
            assert time.perf_counter() - t0 < 20.0
    finally:
        srv.stop()
    assert int(srv.control[_lib.CTRL_STARTED]) == per_sm * sms
    for k in range(0, len(insts), 5):
        r = oracle.tabu_search(oracle.Problem(insts[k], gen.PENALTY, 1000), 6, 80)
        assert int(done[k]["info"][api.INFO_STATUS]) == 0 == r["status"]
        assert int(done[k]["info"][api.INFO_Z_BEST]) == r["z_best"]
        np.testing.assert_array_equal(done[k]["route"][:insts[k].n_missions], r["route"])


def test_two_servers_of_smaller_blocks_share_the_device():
    """Workers of 256 threads leave half of an SM's registers, and shared memory, to another
    launch."""
    servers = [serve.Server(max_loc=40, max_vehicles=10, max_missions=60, n_slots=8) for _ in range(2)]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    inst = gen.random_instance(61, n_loc=40, n_vehicles=8, n_missions=60, duty_cap=500, max_minutes=90)
    try:
        params = api.make_params(6, 50, gen.PENALTY, 1000, block_threads=256)
        torch.cuda.synchronize()
        for srv in servers:  # as Server.start, which first waits for the device
            _lib.check(_lib.load().asched_serve(ctypes.byref(srv.struct), ctypes.byref(params), int(5e9), sms,
                                                ctypes.c_void_p(srv.serve_stream.cuda_stream)), "asched_serve")
            srv.running = True
        for k, srv in enumerate(servers):
            srv.submit(inst, k)
        got, t0 = [None, None], time.perf_counter()
        while any(g is None for g in got) and time.perf_counter() - t0 < 3.0:
            for k, srv in enumerate(servers):
                for slot, _ in srv.poll():
                    got[k] = srv.result(slot)
    finally:
        for srv in servers:
            srv.stop()
    r = oracle.tabu_search(oracle.Problem(inst, gen.PENALTY, 1000), 6, 50)
    for g in got:
        assert g is not None and int(g["info"][api.INFO_Z_BEST]) == r["z_best"]
