#pragma once
// device that holds the address, -1: none
int fake_device_of(const void* p);
// writes a launch down; status: the launch's status word, for the one the test
// has asked to report
void fake_note(const char* what, int* status);
