"""GPU: calls of different sizes from several host threads at once.  A kernel's
limit of dynamic shared memory belongs to the function, so a small call between
a large one's check and its launch must not take the large one's limit away."""
import threading

import numpy as np
import pytest
import torch

import pcv_inputs as pin

pytestmark = pytest.mark.gpu


def together(jobs, rounds):
    """Every job in a thread and stream of its own; the first failure, if any."""
    failed, start = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(rounds):
                    if failed:
                        break
                    job()
                torch.cuda.current_stream().synchronize()
        except Exception as e:          # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return failed


def test_meshes_of_different_sizes():
    from paper_2204_00602_gb300 import autograd as ag
    sets = {m: torch.from_numpy(pin.mesh_phases(1, m * (m - 1), 9960 + m)).cuda() for m in (40, 48, 56, 64)}
    want = {m: ag.mesh_unitary(p, m) for m, p in sets.items()}
    torch.cuda.synchronize()
    assert not together([lambda m=m, p=p: ag.mesh_unitary(p, m) for m, p in sets.items()], 2000)
    for m, p in sets.items():
        assert torch.equal(ag.mesh_unitary(p, m), want[m])


def test_tiles_of_different_sizes():
    import paper_2204_00602_gb300 as pcv
    jobs = []
    for m, n, count in ((128, 5, 64), (60, 4, 300), (100, 3, 40), (128, 4, 200)):
        U, t = torch.from_numpy(pin.haar_unitary(m, 9970)).cuda(), pin.single_photon_input(m, n)
        o = torch.from_numpy(pin.random_outputs(m, n, count, 9971)).cuda()
        jobs.append(lambda U=U, t=t, o=o: pcv.amplitudes(U, t, o, algo=pcv.PCV_ALGO_TILE))
    torch.cuda.synchronize()
    assert not together(jobs, 1000)
