"""Which form of the LM head's product runs: the rules of csrc/lm_forms.h, compiled on their own."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17652_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("lm_forms")
    (d / "r.cc").write_text('#include "lm_forms.h"\n'
                            'extern "C" int pairs(int m, int n, int hidden, int sms) { return fb::lm_pairs(m, n, hidden, sms); }\n'
                            'extern "C" int both(int m, int n, int hidden, int sms) { return fb::lm_both_forms(m, n, hidden, sms); }\n'
                            'extern "C" int masked(int m, int n, int hidden, int sms) {\n'
                            '  return fb::lm_pairs_of(fb::lm_pairs_mask(n, hidden, sms), m);\n'
                            '}\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cc"), "-o", str(d / "r.so")], check=True)
    return ctypes.CDLL(str(d / "r.so"))


# (row tiles, vocabulary tiles, hidden): measured faster that way
@pytest.mark.parametrize("m,n,hidden,form", [
    (0, 592, 2048, 0), (1, 592, 2048, 0), (2, 592, 2048, 1), (3, 592, 2048, 0), (5, 592, 1024, 0), (7, 592, 4096, 0), (11, 592, 1024, 1),
    (13, 592, 2048, 1), (16, 592, 1024, 1), (40, 592, 2048, 1), (41, 592, 2048, 1), (16, 592, 768, 1), (11, 592, 768, 0), (13, 592, 768, 0), (21, 592, 768, 1),
    (13, 91, 4096, 0), (11, 91, 4096, 0), (5, 91, 4096, 1), (1, 64, 2048, 0), (3, 64, 2048, 1), (7, 64, 2048, 1), (9, 64, 2048, 0),
    (131072, 1 << 23, 4096, 1)])
def test_form_by_rounds(rules, m, n, hidden, form):
    assert rules.pairs(m, n, hidden, SMS) == form and rules.masked(m, n, hidden, SMS) == form


def test_mask_holds_the_rule(rules):
    for n in (1, 64, 91, 297, 592):
        for hidden in (768, 2048):
            assert all(rules.masked(m, n, hidden, SMS) == rules.pairs(m, n, hidden, SMS) for m in range(64))
            assert all(rules.masked(m, n, hidden, SMS) == 1 for m in (64, 65, 127, 128, 131072))


# (row tiles of capacity, vocabulary tiles, hidden): where the form that is turned down would cost more than pairs save,
# one form is launched, as where a call is small
@pytest.mark.parametrize("most,n,hidden,both", [
    (3, 592, 4096, 0), (4, 592, 2048, 1), (24, 592, 704, 0), (24, 592, 768, 1), (24, 125, 768, 0), (24, 125, 1024, 1), (8, 250, 1024, 0),
    (8, 250, 2048, 1), (8, 125, 4096, 0), (64, 592, 768, 1), (16, 297, 768, 1), (131072, 1 << 23, 4096, 1)])
def test_both_forms_only_where_pairs_can_pay(rules, most, n, hidden, both):
    assert rules.both(most, n, hidden, SMS) == both and not rules.both(most, n, hidden, 1)


# the live row tiles that test_gpu_lm_pair.py runs at 297 vocabulary tiles and 16 row tiles of capacity, and the contexts that it
# takes for the one-CTA form
def test_forms_of_the_gpu_test(rules):
    tiles = (1, 2, 3, 4, 5, 13, 16)
    assert rules.both(16, 297, 768, SMS) and not rules.both(3, 297, 2048, SMS)
    assert [rules.masked(m, 297, 768, SMS) for m in tiles] == [0, 1, 0, 1, 0, 0, 1]
    assert all([rules.masked(m, 297, h, SMS) for m in tiles] == [0, 1, 0, 1, 0, 1, 1] for h in (1088, 2048))
