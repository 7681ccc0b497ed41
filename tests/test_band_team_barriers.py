"""The shared words of the band kernel's teams, on the CPU: in an ends-free
pair every warp of a team reads the score at which an end was found after a
row's barrier, and the first thread, done with the pair, writes the queue's
next index for the team's broadcast.  Every interleaving of a fast and a slow
warp over these steps, with the words the source uses, gives both warps the
same answer; with one word for both uses it does not."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_02085_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _answers(shared_word, found, last_row, next_index):
    """What the slow warp concludes from its read of the found-score word, over
    every interleaving: after the row's barrier the slow warp reads it once;
    the fast warp reads it and, where the pair is over (an end found, or the
    last row done), writes next_index to the broadcast's word, then waits."""
    over = found or last_row
    out = set()
    row, stale = 7, 0
    for write_first in (False, True):
        word = {"fin": row if found else stale, "slot": -1}
        if over and write_first:
            word["fin" if shared_word else "slot"] = next_index
        out.add(word["fin"] == row)
    return out


def _always_agrees(shared_word):
    return all(_answers(shared_word, found, last, q) == {found}
               for found in (False, True) for last in (False, True) for q in range(12))


def test_one_word_for_both_uses_is_a_race():
    assert not _always_agrees(True)
    assert _always_agrees(False)


def test_found_score_and_broadcast_have_their_own_words():
    pair = re.search(r"band_forward<WPP, CIG, EF>\(.*?bits, &([\w.>-]+), &k_end\)", _read("band_path.cuh"), re.S)
    take = re.search(r"Team<WARPS>::broadcast\(.*?: 0, &([\w.>-]+)\)", _read("band.cu"), re.S)
    assert pair and take
    assert _always_agrees(pair.group(1) == take.group(1)), (pair.group(1), take.group(1))
