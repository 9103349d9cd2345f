"""The life of the pinned words that a decode loop's kernels report to, with the library's calls replaced by fakes."""
import gc
import weakref

import pytest
import torch

from paper_2608_27514_b200 import decode


class _Step:
    S, B, R, k, device = 2, 3, 32, 3, torch.device("cpu")
    status = torch.zeros(1, dtype=torch.int32)
    conf = topk_idx = topk_prob = lse = topk_ws = edge_valid = prefix_len = accepted_node = accepted_len = n_new_tokens = None
    unmask_flag = unmask_tok = None

    def check_status(self):
        pass


@pytest.fixture
def calls(monkeypatch):
    """[(report, ticket)] that kernels have been asked to write, oldest first."""
    seen = []
    zeros = torch.zeros
    monkeypatch.setattr(torch, "zeros", lambda *a, pin_memory=False, **kw: zeros(*a, **kw))
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    monkeypatch.setattr(decode.B, "tsd_begin_block", lambda *a: seen.append((weakref.ref(a[9]) if a[9] is not None else None, a[10])))
    monkeypatch.setattr(decode.B, "tsd_advance_block", lambda *a: seen.append((weakref.ref(a[37]) if a[37] is not None else None, a[34])))
    return seen


def _write(call, masked=0):
    words = call[0]()
    words.fill_(call[1] << 32 | masked)


def test_words_outlive_a_decoder_whose_report_is_in_flight(calls):
    d = decode.BlockDecoder(_Step(), 2, 2, 0.9, 99)
    d.start(torch.zeros(2, 32, dtype=torch.int32))
    d.advance(torch.zeros(1))                       # reports nothing, and does not tell that the first report has arrived
    del d
    gc.collect()
    assert calls[0][0]() is not None                # the kernel that begins the block still has to write there
    _write(calls[0])
    decode.BlockDecoder(_Step(), 2, 2, 0.9, 99)     # the next decoder gives back what has arrived
    gc.collect()
    assert calls[0][0]() is None


def test_words_of_a_report_that_was_seen_are_given_back_at_once(calls, monkeypatch):
    monkeypatch.setattr(decode.B, "tsd_wait_block", lambda report, ticket, stream=None: (0, 0))
    d = decode.BlockDecoder(_Step(), 2, 2, 0.9, 99)
    d.start(torch.zeros(2, 32, dtype=torch.int32))
    d.decode(None)
    del d
    gc.collect()
    assert calls[0][0]() is None


def test_a_rejected_call_leaves_nothing_in_flight(calls, monkeypatch):
    def reject(*a):
        calls.append((weakref.ref(a[9]), a[10]))
        raise decode.B.TsdError(decode.B.TSD_ERR_INVALID_ARG, "tsd_begin_block")
    monkeypatch.setattr(decode.B, "tsd_begin_block", reject)
    d = decode.BlockDecoder(_Step(), 2, 2, 0.9, 99)
    with pytest.raises(decode.B.TsdError):
        d.start(torch.zeros(2, 32, dtype=torch.int32))
    del d
    gc.collect()
    assert calls[0][0]() is None


def test_a_captured_start_reports_nothing(calls, monkeypatch):
    # a graph may be replayed when the decoder is long gone
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    d = decode.BlockDecoder(_Step(), 2, 2, 0.9, 99)
    d.start(torch.zeros(2, 32, dtype=torch.int32))
    assert calls[0][0] is None and not d.begun


def test_words_outlive_a_decoder_dropped_between_two_passes(calls, monkeypatch):
    # the second forward fails while the first pass is still writing its tree: its last word has not arrived
    monkeypatch.setattr(decode.B, "tsd_wait_block", lambda report, ticket, stream=None: (5, 0))
    d = decode.BlockDecoder(_Step(), 2, 2, 0.9, 99)
    d.start(torch.zeros(2, 32, dtype=torch.int32))
    passes = iter([torch.zeros(1)])
    with pytest.raises(StopIteration):
        d.decode(lambda state: next(passes))
    del d
    gc.collect()
    assert calls[1][0]() is not None
    _write(calls[1])
    decode.BlockDecoder(_Step(), 2, 2, 0.9, 99)
    gc.collect()
    assert calls[1][0]() is None
