"""The pair pass keeps the nearest partners as sorted 32-bit words
(csrc/qs_device.cuh: sort4, sort8, merge7). By the 0-1 principle (Knuth, TAOCP
vol. 3, 5.3.4) a network of compare-exchanges and minima is right for every
input iff it is for every one of zeros and ones; this test reads the networks
from the source and checks them all."""
import itertools
import pathlib
import re

SRC = (pathlib.Path(__file__).resolve().parents[1] / "paper_2306_09537_gb300" / "csrc" / "qs_device.cuh").read_text()


def body(signature):
    text = SRC[SRC.index(signature):]
    return text[:text.index("\n}\n")]


def comparators(signature):
    return [(int(a), int(b)) for a, b in re.findall(r"cmp_swap\(\w\[(\d)\], \w\[(\d)\]\)", body(signature))]


def apply(net, seq):
    a = list(seq)
    for i, j in net:
        a[i], a[j] = min(a[i], a[j]), max(a[i], a[j])
    return a


def test_sorting_networks_sort_every_zero_one_input():
    for n, signature in ((4, "void sort4(uint32_t k[4])"), (8, "void sort8(uint32_t k[8])")):
        net = comparators(signature)
        for bits in itertools.product((0, 1), repeat=n):
            assert apply(net, bits) == sorted(bits), (n, bits)


def test_merge_keeps_the_seven_smallest_sorted():
    sig = "void merge7(uint32_t b[7], const uint32_t n[4])"
    minima = [tuple(map(int, m)) for m in re.findall(r"b\[(\d)\] = min\(b\[(\d)\], n\[(\d)\]\)", body(sig))]
    net = comparators(sig)
    assert len(minima) == 4 and len(net) == 9
    for ones_b, ones_n in itertools.product(range(8), range(5)):
        b, n = [0] * (7 - ones_b) + [1] * ones_b, [0] * (4 - ones_n) + [1] * ones_n
        want = sorted(b + n)[:7]
        for to, i, j in minima:
            assert to == i
            b[i] = min(b[i], n[j])
        assert apply(net, b) == want, (ones_b, ones_n)
