"""CPU tests of the host side of libnq's calls, on a faked device (fake_device.cpp):
the request server, whose faked kernel asks of each record what the real one
asks, and what nq_total_ex has searched."""
import os
import subprocess

import pytest

from paper_2511_12009_gb300 import _build, nq, serve

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    nq.lib()  # (built)
    exe = str(tmp_path_factory.mktemp("host") / "fake_device")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", _build.INCLUDE, "-I", _build.CSRC, "-I", cuda,
                    os.path.join(HERE, "fake_device.cpp"), _build.LIB,
                    f"-Wl,-rpath,{_build.OUT_DIR}", "-o", exe], check=True)

    def run(*args):
        return subprocess.run([exe] + [str(a) for a in args], check=True, capture_output=True,
                              text=True, timeout=120).stdout.strip()
    return run


def test_every_cut_is_one_the_kernel_takes(host):
    """serve_cut over all boards, depths and stacks, the widest index (31 bits) among
    them: the kernel takes each cut, and a digit covers its row's columns."""
    made, wide, refused, short = (int(x.split()[0]) for x in host("cuts").split(", "))
    assert made > 100000 and wide > 1000
    assert refused == 0 and short == 0


def test_every_shape_that_fits_is_planned(host):
    """Launch shapes up to the last bytes of an SM's shared memory."""
    fit, refused = (int(x.split()[0]) for x in host("shapes").split(", "))
    assert fit > 100000 and refused == 0


@pytest.mark.parametrize("max_n,stack,n,queens", [
    (21, 9, 21, []), (21, 9, 21, [16, 15, 19, 6]), (22, 9, 22, [19, 20, 13, 5, 16, 6]),
    (26, 0, 26, [15, 18, 14, 1, 2, 10, 20, 4, 17, 14]), (18, 4, 18, []), (20, 0, 20, [])])
def test_admitted_requests_are_searched(host, max_n, stack, n, queens):
    """Requests whose records are cut 31 bits wide (all but the last) are admitted
    with records that the kernel searches, every one."""
    records, first, second = host("burst", max_n, stack, n, *queens).split(", ")
    assert first == f"poll 0: answer {records.split()[0]}" and second == "poll 0:"


def test_a_request_not_searched_whole_has_no_count(host):
    """A record that the kernel gives back unsearched is an error, and what the others
    found is not delivered as the request's count."""
    _, first, second = host("refuse", 20, 0, 12, 3, 4).split(", ")
    assert first == f"poll {nq.NQ_EINVAL}: answer {serve.NO_COUNT}" and second == "poll 0:"


def test_poll_keeps_what_finished_beside_an_error(monkeypatch):
    """Answers that nq_server_poll hands over together with an error come with the next
    poll of the Python server."""
    class Lib:
        polls = [(nq.NQ_EINVAL, [(1, 10), (2, serve.NO_COUNT)]), (nq.NQ_OK, [(3, 30)])]

        def nq_server_poll(self, h, tickets, counts, size, got):
            rc, done = self.polls.pop(0)
            for i, (t, c) in enumerate(done):
                tickets[i], counts[i] = t, c
            got._obj.value = len(done)
            return rc

        nq_server_create = nq_server_destroy = staticmethod(lambda *a: nq.NQ_OK)
        nq_strerror = nq.lib().nq_strerror

    lib = Lib()
    monkeypatch.setattr(nq, "lib", lambda: lib)
    monkeypatch.setattr(serve, "_declare", lambda: lib)
    srv = serve.Server()
    with pytest.raises(nq.NQError):
        srv.poll()
    assert srv.poll() == [(1, 10), (2, None), (3, 30)]


@pytest.mark.parametrize("n,d", [(12, 6), (13, 2), (14, 5), (16, 6), (9, 9), (8, 1)])
def test_total_searches_the_depth_that_is_asked_for(host, n, d):
    """A chosen depth is the depth of the records that are searched, and the one timed."""
    m = nq.prefix_count(n, d)
    assert host("total", n, d) == (f"search {m} records of {d} rows, rc 0, total {m}, "
                                   f"timing {m} of {d}")


@pytest.mark.parametrize("n", [3, 5, 12, 16])
def test_total_chooses_four_rows(host, n):
    """With no depth given the default form searches at most four rows' prefixes; the
    timing is of the default depth's set."""
    d = nq.default_depth(n)
    m = nq.prefix_count(n, min(d, 4))
    want = f"search {m} records of {min(d, 4)} rows, " if m else ""
    assert host("total", n, 0) == (want + f"rc 0, total {m}, "
                                   f"timing {nq.prefix_count(n, d)} of {d}")


def test_a_failed_host_allocation_does_not_end_the_process(host):
    """Whichever host allocation of a synchronous call fails, its clean-up does not throw;
    planning a launch needs none."""
    calls, codes = host("nomem").split(", ")[-2:]
    assert int(calls.split()[0]) >= 3 and codes == "count 0 0 0"
