// The status that an asynchronous call's kernel leaves in host memory: reported once, with its message.
// Exits 0 when all holds.  Built against the library by test_late_status.py.
#include <cstdio>
#include <cstring>

#include "internal.h"

using namespace qs;

int main() {
  State st;
  if (late_status(&st) != QS_OK) return 1;   // no such call yet
  int word = 0;
  st.late = &word;
  if (late_status(&st) != QS_OK) return 2;
  word = QS_ETIMEOUT;
  if (late_status(&st) != QS_ETIMEOUT || !std::strstr(qs_last_error(), "bounded wait")) return 3;
  if (word != 0 || late_status(&st) != QS_OK) return 4;
  word = QS_EUNSUPPORTED;
  if (late_status(&st) != QS_ECUDA || late_status(&st) != QS_OK) return 5;
  return 0;
}
