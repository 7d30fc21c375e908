"""The order in which a step issues its casts and GEMM batches on the two streams, on stand-ins for the streams (no GPU)."""
import contextlib

import pytest
import torch

from paper_2511_23225_b200 import workload


class Stream:
    def __init__(self, log, name):
        self.log, self.name = log, name

    def wait_stream(self, other):
        self.log.append((self.name, "wait", other.name))

    def wait_event(self, ev):
        self.log.append((self.name, "wait", ev.at))


class Event:
    def record(self, stream):
        self.at = (stream.name, len([e for e in stream.log if e[0] == stream.name and e[1] != "wait"]))


@pytest.fixture
def issue(monkeypatch):
    def run(variant, linears):
        log, current = [], []
        main, side = Stream(log, "main"), Stream(log, "side")

        @contextlib.contextmanager
        def on(s):
            current.append(s)
            yield
            current.pop()

        monkeypatch.setattr(torch.cuda, "current_stream", lambda: main)
        monkeypatch.setattr(torch.cuda, "stream", on)
        monkeypatch.setattr(torch.cuda, "Event", Event)
        b = object.__new__(workload.BlockStep)
        b.variant, b.overlap, b.side, b.M, b.linears = variant, True, side, 512, list(range(linears))
        b.group_ok = lambda lb: True
        name = lambda: (current[-1] if current else main).name
        b.quantize_all = lambda lbs: log.append((name(), "cast", tuple(lbs)))
        b.run_gemm_batch = lambda batch: log.append((name(), "gemm", tuple(batch)))
        b.tweo = lambda: log.append((name(), "loss"))
        b.update_output_scales = lambda: log.append((name(), "scales"))
        b.step()
        return log
    return run


def kinds(log):
    return [e[1] for e in log if e[1] in ("cast", "gemm", "loss")]


@pytest.mark.parametrize("variant", ["plain", "fused"])
def test_all_casts_and_the_loss_go_before_the_first_gemm_and_wait_for_none(issue, variant):
    log = issue(variant, 5)
    assert kinds(log) == ["cast"] * 3 + ["loss"] + ["gemm"] * 3
    assert [e for e in log if e[0] == "side" and e[1] == "wait"] == [("side", "wait", "main")]


def test_without_the_fused_epilogue_a_gemm_batch_goes_ahead_of_the_next_casts(issue):
    log = issue("unfused", 5)
    assert kinds(log) == ["cast", "gemm", "cast", "gemm", "cast", "gemm", "loss"]


@pytest.mark.parametrize("variant", workload.VARIANTS)
@pytest.mark.parametrize("linears", [1, 2, 4, 5])
def test_every_gemm_batch_waits_for_its_casts_and_the_step_for_both_streams(issue, variant, linears):
    log = issue(variant, linears)
    casts = [e[2] for e in log if e[1] == "cast"]
    for at, e in enumerate(log):
        if e[1] != "gemm":
            continue
        needed = max(i for i, c in enumerate(casts) if set(c) & set(e[2])) + 1     # side-stream operations to be over
        waits = [w[2] for w in log[:at] if w[0] == "main" and w[1] == "wait"]
        assert any(w[0] == "side" and w[1] >= needed for w in waits)
    assert log[-1] == ("main", "wait", "side") and ("main", "scales") in log
