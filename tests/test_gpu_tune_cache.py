"""The autotuner's cache file across changes of what its variant numbers mean."""
import pytest

from paper_1405_6104_gb300 import binding as B
from paper_1405_6104_gb300 import systems as S

pytestmark = pytest.mark.gpu


def test_entries_of_an_earlier_meaning_are_tuned_anew(tmp_path):
    """A file from before the variants were renumbered (a key without a
    version): its choice is not taken, a new entry is added and serves from
    then on."""
    from paper_1405_6104_gb300 import build
    build.build()
    s, p = S.tiny_chain(0)
    cache = tmp_path / "tune.txt"
    old = "a8_t0_d1_nt1 2 2\n"  # 212 atoms, one trial, 7.9 atoms per nm^3, one type
    cache.write_text(old)
    with B.TrialBatch(s, p, [1]) as b:
        first = B.sim_autotune(b.h, 1, str(cache))
        text = cache.read_text()
        assert text.startswith(old) and len(text.splitlines()) == 2
        key, pv, cv = text.splitlines()[1].split()
        assert (int(pv), int(cv)) == first and key != old.split()[0]
    with B.TrialBatch(s, p, [1]) as b:
        assert B.sim_autotune(b.h, 1, str(cache)) == first
    assert cache.read_text() == text
