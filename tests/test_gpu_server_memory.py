"""A served job that the device cannot hold beside the others, though the budget admits
it, waits for their memory instead of failing (GPU only; the shortage is an allocator
that refuses above a limit)."""
import pytest

from synthetic import add_walls, phi0_blob, sphere_pack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fit", [1.5, 2.5])     # jobs that the limit holds at once
def test_job_waits_for_memory(fit, monkeypatch):
    import paper_2007_12266_gb300 as lbm
    live, peak, limit = {}, [0], [float("inf")]
    real = lbm._torch_allocator

    def limited(torch, device, stream):
        alloc, free = real(torch, device, stream)

        def _alloc(nbytes, strm, user):
            if sum(live.values()) + nbytes > limit[0]:
                return 0
            p = alloc(nbytes, strm, user)
            if p:
                live[p] = nbytes
                peak[0] = max(peak[0], sum(live.values()))
            return p

        def _free(ptr, user):
            live.pop(ptr, None)
            free(ptr, user)
        keep.append((alloc, free))
        return lbm._lib.ALLOC_FN(_alloc), lbm._lib.FREE_FN(_free)
    keep = []
    monkeypatch.setattr(lbm, "_torch_allocator", limited)
    lab = add_walls(sphere_pack((48, 48, 48), 0.35, 5.0, 1.0, 3).labels, ("x", "y"))
    phi0 = phi0_blob(lab, 0.4, 5)
    s = lbm.Server(max_jobs=4, check_interval=10)

    def run(n):
        tickets = [s.submit(lab, phi0, None, kind="steady", max_steps=20, periodic=(0, 0, 1),
                            force=(0, 0, 1e-5)) for _ in range(n)]
        most = 0
        for _ in range(100):
            running, queued, _ = s.run()
            most = max(most, running)
            if running == 0 and queued == 0:
                break
        return tickets, most
    tickets, _ = run(1)                          # one job's memory
    assert s.poll(tickets[0])["state"] == "done"
    s.release(tickets[0])
    limit[0] = fit * peak[0]
    tickets, most = run(4)
    assert [s.poll(t)["state"] for t in tickets] == ["done"] * 4
    assert most <= fit
    s.close()
