"""Chained launches wait for whatever precedes them on their stream: foreign kernels and copies between the library's calls, and
other streams joined by events, order as they do between ordinary launches."""
import numpy as np
import pytest

from paper_2402_04514_gb300 import assembly, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,degree", [((11, 9), 1), ((160, 150), 2)])
def test_foreign_work_between_calls(cells, degree):
    """Each round changes the state by a kernel or a copy of torch's, on the same stream or on another one that waits for the
    library's last call and is waited for by its next: the bits of the same rounds with a synchronisation between any two."""
    import torch

    from paper_2402_04514_gb300.gdg import Solver

    P = assembly.assemble_2d(*cells, degree)
    U0 = torch.from_numpy(workloads.four_quadrant(P.x[0], P.x[1], seed=1)).cuda()
    S = Solver(P)
    S.set_clock(0.0, float("inf"), 0.3)

    def rounds(sync):
        S.set_clock(0.0, float("inf"), 0.3)
        main, side = torch.cuda.Stream(), torch.cuda.Stream()
        U, work, V, outs = U0.clone(), (torch.empty_like(U0), torch.empty_like(U0)), torch.empty_like(U0), []
        torch.cuda.synchronize()

        def wait():
            if sync:
                torch.cuda.synchronize()

        for k in range(12):
            with torch.cuda.stream(main):
                S.step(U, work, stream=main)
                wait()
                if k % 3 == 0:
                    U.mul_(1.0 + 2.0 ** -10)  # a kernel in between
                elif k % 3 == 1:
                    V.copy_(U)  # a copy out, a change, a copy in
                    V.mul_(1.0 - 2.0 ** -11)
                    U.copy_(V)
                wait()
            if k % 3 == 2:
                side.wait_event(main.record_event())
                with torch.cuda.stream(side):
                    V.copy_(U)
                    U.add_(V, alpha=2.0 ** -12)
                    wait()
                main.wait_event(side.record_event())
            with torch.cuda.stream(main):
                outs.append(U.clone())
                wait()
        torch.cuda.synchronize()
        return outs

    want = rounds(True)
    for _ in range(3):
        for k, (a, b) in enumerate(zip(rounds(False), want)):
            assert torch.equal(a, b), k
