"""A served job whose device waits ran out fails alone (fake backend, no GPU)."""
import test_serve_host as host

from paper_1710_05155_gb300 import serve


class Backend(host.FakeBackend):
    def failure(self, jid):
        return "KA_ETIMEOUT" if self.jobs[jid][0].tag["index"] == 1 else ""


def test_a_job_without_a_result_fails_alone():
    clock = host.FakeClock()
    be = Backend(clock)
    server = serve.Server(be, clock=clock, sleep=clock.sleep, autotune=False, keep_results=True)
    report = server.run([host.job(i, 0.0, 20, 10) for i in range(3)])
    assert [r.status for r in server.records] == ["done", "failed", "done"]
    assert report["done"] == 2 and report["failed"] == 1
    assert server.records[1].counts is None and server.records[1].error == "KA_ETIMEOUT"
    assert not be.jobs  # its memory is given back too
