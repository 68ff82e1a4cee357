"""The rule that splits the scoring of few long events among CTAs: only where some CTA's share becomes shorter, and not for the
calls that were measured slower for it."""
import pytest

from akv_split import prefill_split, prefill_tail, prefill_tail_split, split_share


@pytest.mark.parametrize("sms", [148, 132, 80])
@pytest.mark.parametrize("topk", [False, True])
@pytest.mark.parametrize("ragged", [False, True])
def test_a_split_shortens_every_share(sms, topk, ragged):
    for events in (1, 2, sms // 5, sms * 2 // 9, sms // 4, sms // 4 + 1, sms * 4 // 9, sms // 2, sms // 2 + 1, sms - 1, sms, sms + 1, 4 * sms):
        for N in list(range(257, 5121, 61)) + [1023, 1024, 1025, 2047, 2048, 2049, 3072, 3073, 5120]:
            split, stages = prefill_split(events, N, sms, topk, ragged), (N + 63) // 64
            assert split in (1, 2, 4)
            if split == 1:
                continue
            assert events <= sms and split_share(stages, split) * 4 <= stages * 3
            if split * events > 2 * sms or (split == 2 and 2 * events > sms):   # more than a pair on an SM, or a pair without two to a cluster
                assert not ragged and split == 2 and split_share(stages, 2) <= 0.516 * stages


# (events, rows, top-k, ragged, how many CTAs): 148 multiprocessors; the calls that a split made slower take one CTA per event
@pytest.mark.parametrize("events,N,topk,ragged,split", [
    (112, 2113, True, False, 1), (112, 2048, True, False, 1), (148, 2560, True, False, 1), (112, 3136, True, False, 1),   # top-k
    (37, 1100, True, False, 1), (74, 4096, True, False, 2), (74, 4096, False, False, 2),
    (112, 2113, False, False, 1), (148, 2113, False, False, 1), (112, 3136, False, False, 1), (112, 3904, False, False, 1),   # a share that is hardly shorter
    (112, 4096, True, True, 1), (148, 4096, False, True, 1),   # candidate counts unknown
    (160, 4096, False, False, 1), (896, 4096, False, False, 1), (28, 900, False, False, 1),
    (112, 5000, False, False, 2), (112, 4096, False, False, 2), (148, 3072, False, False, 2), (112, 3072, True, False, 2),
    (28, 4096, False, False, 4), (28, 1100, True, False, 4), (37, 1100, False, False, 4), (56, 4096, False, True, 4), (74, 2049, True, False, 2)])
def test_calls_that_were_measured(events, N, topk, ragged, split):
    assert prefill_split(events, N, 148, topk, ragged) == split


# (events, rows, top-k, ragged, how many of them are left to a second launch): 148 multiprocessors, 296 places
@pytest.mark.parametrize("events,N,topk,ragged,tail", [
    (896, 4096, True, False, 8), (896, 4096, False, False, 0), (304, 3072, True, False, 8), (304, 2113, True, False, 0), (370, 5000, True, False, 74),
    (371, 4096, True, False, 0), (296 + 112, 3136, True, False, 0), (592, 4096, True, False, 0), (296, 4096, True, False, 0), (8, 4096, True, False, 0),
    (304, 4096, True, True, 0), (296 + 148, 4096, True, False, 0), (296 + 200, 4096, True, False, 0)])
def test_events_left_to_a_second_launch(events, N, topk, ragged, tail):
    assert prefill_tail(events, N, 148, topk, ragged) == tail
    if tail:
        assert prefill_split(tail, N, 148, topk, ragged) > 1


@pytest.mark.parametrize("sms", [148, 132, 80])
def test_ctas_that_share_a_last_event_have_an_sm_each(sms):
    for rest in range(1, 2 * sms):
        tail = prefill_tail(2 * sms + rest, 4096, sms, topk=True)
        if tail:
            split = prefill_tail_split(tail, sms)
            assert tail == rest and split in (2, 4) and tail * split <= sms
            assert split == 4 or tail * 4 > sms
