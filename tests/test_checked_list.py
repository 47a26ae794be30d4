"""CPU check of the checked build's index tests in the wide row form: the
function that turns an entry of the connected list into a configuration,
compiled for the host with the checks on and run on lists with entries out of
range. No GPU work is issued."""

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), 'paper_2204_07816_gb300', 'csrc')

PROGRAM = r'''
#include <cstdio>
#include <cstdlib>
#define __device__
#define NQS_INDEX_OK(cond, err) ((cond) ? true : ((*(err) |= 1), false))
#include "wide_list.cuh"
int main(int argc, char **argv) {
    const int16_t ci[4] = {3, 15, -1, 5}, cj[4] = {7, 0, 2, 16};
    int err = 0;
    const nqs::WideCfg c = nqs::wide_entry(ci, cj, atoi(argv[1]), 4, 16, &err);
    printf("%d %d %d %d\n", c.i, c.j, c.roll, err);
}
'''


@pytest.fixture(scope='module')
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp('wide_list')
    (d / 'main.cpp').write_text(PROGRAM)
    subprocess.run(['g++', '-std=c++17', '-I', CSRC, '-o', str(d / 'main'), str(d / 'main.cpp')], check=True)
    return str(d / 'main')


@pytest.mark.parametrize('k,want', [(0, '3 7 0 0'), (1, '15 0 0 0'), (2, '-1 -1 0 1'), (3, '-1 -1 0 1'), (4, '-1 -1 0 1'),
                                    (-1, '-1 -1 0 1'), (40000, '-1 -1 0 1')])
def test_list_entry_out_of_range_is_reported_and_not_used(program, k, want):
    assert subprocess.run([program, str(k)], capture_output=True, text=True, check=True).stdout.strip() == want


def test_the_wide_form_reads_the_list_through_the_check():
    """No other line of the wide form reads the list's sites; the log psi list is indexed after a check."""
    text = open(os.path.join(CSRC, 'tc.cu')).read()
    wide = text[text.index('wide row form\n// The row form with'):text.index('// ---------------------------------------------------------------- kernel prologue')]
    reads = [l for l in wide.splitlines() if 'ord[' in l and 'e.ord[k] =' not in l and 'e.ord[base + off] =' not in l]
    # e.ord: every read goes through wide_entry, or is the index that the next check tests
    assert reads and all('wide_entry(' in l or 'idx = q < 0 ? 0 : e.ord[q] + lead' in l for l in reads)
    assert 'NQS_INDEX_OK(idx >= 0 && idx < n_entries, err)' in wide
