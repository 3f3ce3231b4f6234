// tune_file_check.cpp -- reads a file of timed y-pass forms (tune_file.h) for one
// digest and writes what it took of it to a second file for another.  Built and
// run by tests/test_tune_file_host.py.
// Arguments: file, digest, second file, second digest.
#include <stdlib.h>

#include "tune_file.h"

int main(int, char **argv)
{
    isofft::TuneMap m;
    isofft::tune_file_read(argv[1], strtol(argv[2], 0, 0), 3, m);
    isofft::tune_file_write(argv[3], strtol(argv[4], 0, 0), m);
    return 0;
}
