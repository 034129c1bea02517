"""Calls of several host threads: each handle is its own, the kernels' launch
limits are shared by the process."""
import threading

import numpy as np
import pytest

from paper_1711_10579_gb300 import cases

torch = pytest.importorskip("torch")


def mesh(n):
    return cases.transmission_case(n, int(1.35 * n), n // 5, 1, max_angle=0.06)


@pytest.mark.gpu
@pytest.mark.parametrize("prec,B", [("fp64", 1), ("mixed", 1), ("mixed", 320)])
def test_solves_of_two_sizes_from_two_threads(prec, B):
    """A larger and a smaller grid solved by the same kernel from two threads, a
    third thread creating cases: every call is launched (a launch whose shared
    memory exceeds a limit set by another thread would be refused)."""
    import __graft_entry__

    __graft_entry__.build()
    from paper_1711_10579_gb300 import pf

    errors = []
    stop = threading.Event()

    def solve(n, count):
        try:
            ctx = pf.pf_ctx_create(0)
            case = mesh(n)
            c = pf.pf_create_case(ctx, case)
            ld = [torch.tensor(a, device="cuda") for a in cases.scenario_loads(case, B, seed=1)]
            vm, va = (torch.zeros((B, n), dtype=torch.float64, device="cuda") for _ in range(2))
            info = torch.zeros((B, pf.INFO_DTYPE.itemsize), dtype=torch.uint8, device="cuda")
            o = pf.make_opts(precision=pf.PF_FP64 if prec == "fp64" else pf.PF_MIXED)
            for _ in range(count):
                pf.pf_solve_batch_device(c, B, *ld, o, vm, va, info, 0)
            torch.cuda.synchronize()
            got = np.frombuffer(info.cpu().numpy().tobytes(), dtype=pf.INFO_DTYPE)
            if not np.all(got["status"] == 0):
                errors.append((n, got["status"]))
            pf.pf_destroy_case(c)
            pf.pf_ctx_destroy(ctx)
        except Exception as e:  # the assertion below reports it
            errors.append((n, repr(e)))

    def create():
        try:
            ctx = pf.pf_ctx_create(0)
            case = mesh(60)
            while not stop.is_set():
                pf.pf_destroy_case(pf.pf_create_case(ctx, case))
            pf.pf_ctx_destroy(ctx)
        except Exception as e:
            errors.append(("create", repr(e)))

    count = 4000 if B == 1 else 600
    threads = [threading.Thread(target=solve, args=a) for a in ((800, count), (410, count))]
    maker = threading.Thread(target=create)
    for t in (*threads, maker):
        t.start()
    for t in threads:
        t.join()
    stop.set()
    maker.join()
    assert not errors
