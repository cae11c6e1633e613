"""When the request loop holds a request back so that others may join it
(hough_gather.h, host only): not while a client waits for its results or
collects them, not a full batch and not a lone request; requests that keep
coming while nobody looks are gathered."""
import os
import subprocess

import pytest

from paper_2511_02742_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    exe = tmp_path_factory.mktemp("gather") / "gather"
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-I",
                    os.path.join(build.PKG, "csrc"), os.path.join(HERE, "c", "gather.cpp"),
                    "-o", str(exe)], check=True)

    def f(slots, slot_windows, request_windows, clients, gap_us, requests):
        r = subprocess.run([str(exe)] + [str(x) for x in (slots, slot_windows, request_windows,
                                                          clients, gap_us, requests)],
                           check=True, capture_output=True, text=True)
        batches, largest, waited_ns = (int(x) for x in r.stdout.split())
        return batches, largest, waited_ns
    return f


@pytest.mark.parametrize("slots,clients", [(2, 1), (2, 2), (4, 2), (4, 4), (16, 8)])
def test_clients_that_wait_for_their_results(run, slots, clients):
    assert run(slots, 256, 20, clients, 0, 2000)[2] == 0


@pytest.mark.parametrize("gap_us", [5, 20, 39, 55])
def test_results_that_are_collected_at_once(run, gap_us):
    assert run(4, 256, 20, 0, gap_us, 600)[2] == 0


@pytest.mark.parametrize("slots", [2, 4, 16])
def test_requests_that_keep_coming_unread_are_gathered(run, slots):
    batches, largest, waited = run(slots, 256, 20, -1, 39, 60)
    assert largest >= 2 and batches <= 45, (batches, largest, waited)
    assert 0 < waited <= 60_000


@pytest.mark.parametrize("slots", [2, 16])
def test_lone_requests_start_at_once(run, slots):
    assert run(slots, 256, 20, -1, 60, 200) == (200, 1, 0)


@pytest.mark.parametrize("slot_windows,request_windows", [(64, 64), (64, 100), (200, 152), (1, 1)])
def test_a_full_batch_starts_at_once(run, slot_windows, request_windows):
    batches, largest, waited = run(8, slot_windows, request_windows, -1, 15, 400)
    assert waited == 0 and largest == 1


def test_requests_without_windows(run):
    batches, largest, waited = run(4, 64, 0, -1, 10, 300)
    assert largest > 1 and waited <= 60_000
