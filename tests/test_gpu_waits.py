"""Waits of many host threads: each thread steps a bed of its own on a stream
of its own and waits for the sums of every call.  Only a few of the waits may
poll without sleeping, so as many threads as the host has cores keep less than
half of the cores busy while the GPU works."""
import os
import threading
import time

import pytest
import torch

from paper_1111_1129_gb300 import LBMState, SparseLattice, build, capi, inputs, omega_minus

pytestmark = pytest.mark.gpu

WP = 1.0 / 0.8


def test_waiting_threads_leave_the_cores_free():
    build.build()
    capi.load()
    cores = len(os.sched_getaffinity(0))
    if cores < 8:
        pytest.skip("needs eight cores")
    bed = inputs.bed_small(0)
    flags = torch.from_numpy(bed.flags).cuda()
    torch.cuda.synchronize()
    gate = threading.Barrier(cores + 1)
    flux = []

    def work():
        with torch.cuda.stream(torch.cuda.Stream()):
            lat = SparseLattice(flags, "lex", periodic=bed.periodic)
            st = LBMState(lat, "f32s")
            st.step(400, WP, omega_minus(WP), (0.0, 0.0, 1e-6))
            st.reduce_flux(2)
            gate.wait()
            for _ in range(100):
                st.step(400, WP, omega_minus(WP), (0.0, 0.0, 1e-6))
                last = st.reduce_flux(2)
            gate.wait()
            flux.append(last)
            st.close()
            lat.close()

    threads = [threading.Thread(target=work) for _ in range(cores)]
    for t in threads:
        t.start()
    gate.wait()
    wall, cpu = time.perf_counter(), time.process_time()
    gate.wait()
    wall, cpu = time.perf_counter() - wall, time.process_time() - cpu
    for t in threads:
        t.join()
    assert len(flux) == cores and len(set(flux)) == 1
    assert cpu <= 0.5 * cores * wall, (cpu / wall, cores)
