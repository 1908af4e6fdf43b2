"""The chaining of launches across streams, on a fake runtime."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("order") / "check")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-o", out, os.path.join(HERE, "launch_order_check.cpp")], check=True)
    return lambda script: subprocess.run([out] + script.split(), capture_output=True, text=True, check=True, timeout=60).stdout.splitlines()


def test_a_call_on_another_stream_waits_for_the_last_one(check):
    assert check("call 1 call 1 call 2") == ["launch stream 1", "record event 1 stream 1", "status 0",
                                             "launch stream 1", "record event 1 stream 1", "status 0",
                                             "wait stream 2 event 1", "launch stream 2", "record event 1 stream 2", "status 0"]


def test_a_captured_call_neither_waits_nor_records(check):
    got = check("call 1 capture 2 call 2 end call 3")
    assert got[3:5] == ["launch stream 2", "status 0"]
    # the calls after it are chained to the last one outside the capture
    assert got[5:] == ["wait stream 3 event 1", "launch stream 3", "record event 1 stream 3", "status 0"]


def test_a_call_that_failed_half_way_is_waited_for(check):
    # the kernels it had queued before the error are on the stream
    assert check("fail 1 call 2") == ["launch stream 1", "record event 1 stream 1", "status -5",
                                      "wait stream 2 event 1", "launch stream 2", "record event 1 stream 2", "status 0"]


def test_devices_do_not_wait_for_each_other(check):
    # the launch on one device waits (up to ten seconds) for one on the other to begin, in another thread
    assert check("both 0 both 1") == ["both launches at once"] * 2
